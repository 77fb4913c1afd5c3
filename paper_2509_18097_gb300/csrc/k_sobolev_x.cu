// x passes of the grid Sobolev preconditioner (Sec. 3.2, Eq. 3) by line transforms
// (sobolev_line.cuh) and the Adam update (Sec. 3.6):
//   x forward   DCT-II of the x-lines                                 g -> tmp
//   x inverse   of tmp, then Adam on theta, m, v of those vertices
// A tile is XL neighbouring x-lines of three channels, so that the update owns whole float4
// values of theta.  Elements of a line are contiguous in memory: lanes run along the line in
// the loads and stores and along the pairs in the transform stages; the shared rows are padded by
// one pair, which leaves two lanes to a bank in the former and none shared in the latter.
//
// What bounds them: at 256^3 the forward pass takes 67 us inside a frame (planes away from the
// points are skipped) and 138 us on a dense gradient (403 MB, 60 us at the copy rate; L1 and shared
// memory are 77% busy), the inverse with Adam 328 us (1.5 GB, 222 us); a warp-per-line
// FFT with one-channel tiles, whose update touched theta in 4-byte strides, took 500 and about 1200.
// 56 registers (3 blocks per SM) beat 80 (147 and 162 against 141 and 145 us on a dense gradient);
// prefetching the moments and theta to L2 before the transform (388 us), two vertices per thread
// at a time (338) and 64-bit indices (340) did not help the update.
#include "sobolev_line.cuh"

namespace pdg {

constexpr int X_THREADS = 384, X_WARPS = X_THREADS / 32;

template <int n>
struct XT {
  static constexpr int XL = x_lines(n), H = XL / 2, P = 3 * H, S = P + 1, nl = n * n, STEP = X_THREADS / P;
  static_assert(X_THREADS % P == 0 && Fac<n>::N1 <= STEP, "one stage 1 item per thread");
  // float index of row r (position or frequency) of line l, channel c
  static __device__ __forceinline__ int at(int r, int c, int l) { return 2 * (r * S + c * H + (l >> 1)) + (l & 1); }
};

// the n values of a line (zeros if !in) to put(e, value), all of a lane's loads before any use
template <int n, class Put>
__device__ __forceinline__ void line_load(const float* __restrict__ src, bool in, int lane, Put put) {
  constexpr int U = (n + 31) / 32;
  float x[U];
#pragma unroll
  for (int u = 0; u < U; ++u) x[u] = in && lane + 32 * u < n ? src[lane + 32 * u] : 0.f;
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (lane + 32 * u < n) put(lane + 32 * u, x[u]);
}

constexpr int x_smem(int n) { return n * (3 * (x_lines(n) / 2) + 1) * 8; }

// x forward
template <int n>
__device__ __forceinline__ void x_fwd(const Job& J, const Level& lv, int tile, float2* smem, int2 zr) {
  using L = XT<n>;
  constexpr int P = L::P, S = L::S, STEP = L::STEP, XL = L::XL, nl = L::nl, N1 = Fac<n>::N1, N2 = Fac<n>::N2;
  const int r0 = tile * XL, tid = thread_here(), lane = tid & 31, warp = tid >> 5;
  // outside the active planes the tile is zero: not written, read as zero by the passes after
  if (min(r0 + XL - 1, nl - 1) / n < zr.x || r0 / n >= zr.x + zr.y) return;
  float* f = reinterpret_cast<float*>(smem);
  float2* sm = smem + tid % P;
  const int it0 = tid / P;
  if (J.ext_in) {  // a caller's gradient, [n^3][3]: the tile is one contiguous range
    const float* src = J.ext_in + (size_t)r0 * n * 3;
#pragma unroll 1
    for (int l = warp; l < XL; l += X_WARPS)
      line_load<3 * n>(src + (size_t)l * 3 * n, r0 + l < nl, lane,
                       [&](int i, float x) { f[L::at(i / 3, i - i / 3 * 3, l)] = x; });
  } else {
    const float* src = lv.g + (size_t)r0 * n;
#pragma unroll 1
    for (int r = warp; r < 3 * XL; r += X_WARPS) {  // a warp per line
      const int c = r / XL, l = r - c * XL;
      const bool in = r0 + l < nl && (unsigned)((r0 + l) / n - zr.x) < (unsigned)zr.y;
      line_load<n>(src + (size_t)c * lv.n3 + l * n, in, lane, [&](int e, float x) { f[L::at(e, c, l)] = x; });
    }
  }
  __syncthreads();
  {
    float2 v[N2];
    const int s = min(it0, N1 - 1);  // threads without an item load another's: v is always defined
#pragma unroll
    for (int m = 0; m < N2; ++m) v[m] = sm[esrc<n>(s, m) * S];
    __syncthreads();  // the stage writes other rows than it reads
    if (it0 < N1) fwd_stage1<n, S>(v, sm, it0, lv.twm);
  }
  __syncthreads();
  fwd_stage2<n, S, STEP>(sm, it0);
  __syncthreads();
#pragma unroll 1
  for (int q = it0; q < n / 2 + 1; q += STEP) {
    const int nq = q ? n - q : 0;
    float2 xq, xn;
    dct2_ends(sm[q * S], sm[nq * S], __ldg(lv.tw4 + q), xq, xn);
    sm[q * S] = xq;
    if (q && 2 * q != n) sm[nq * S] = xn;
  }
  __syncthreads();
  float* dst = lv.tmp + (size_t)r0 * n;
#pragma unroll 1
  for (int r = warp; r < 3 * XL; r += X_WARPS) {
    const int c = r / XL, l = r - c * XL;
    if (r0 + l < nl)
      for (int k = lane; k < n; k += 32) dst[(size_t)c * lv.n3 + l * n + k] = f[L::at(k, c, l)];
  }
}

// Adam (PyTorch semantics) on the tile's vertices with the gradient in f
template <int n>
__device__ __forceinline__ void adam_tile(const Job& J, const Level& lv, int r0, int tid, const float* f) {
  using L = XT<n>;
  const int cnt = min(L::XL, L::nl - r0) * n;
  const int n3 = lv.n3, v0 = r0 * n;
  const float b1 = J.beta1, b2 = J.beta2, eps = J.eps;
  const float step = lv.lr * J.bias[0], ib2 = J.bias[1];
  const bool pre = J.precondition, keep = J.keep_pgrad && pre;
  float* mp = lv.m + v0;
  float* vp = lv.v + v0;
  float4* th = lv.theta + (size_t)r0 * n;
#pragma unroll 1
  for (int v = tid; v < cnt; v += X_THREADS) {
    const int l = v / n, e = v - l * n;
    float m[3], s[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      m[c] = mp[c * n3 + v];
      s[c] = vp[c * n3 + v];
    }
    float4 t = th[v];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float g = pre ? f[L::at(e, c, l)] : lv.g[v0 + c * n3 + v];
      m[c] = b1 * m[c] + (1.f - b1) * g;
      s[c] = b2 * s[c] + (1.f - b2) * g * g;
      (&t.x)[c] -= step * m[c] / (sqrtf(s[c]) * ib2 + eps);
      mp[c * n3 + v] = m[c];
      vp[c * n3 + v] = s[c];
      if (keep) lv.tmp[v0 + c * n3 + v] = g;
    }
    th[v] = t;
  }
}

// x inverse, then Adam
template <int n>
__device__ __forceinline__ void x_inv(const Job& J, const Level& lv, int tile, float2* smem) {
  using L = XT<n>;
  constexpr int P = L::P, S = L::S, STEP = L::STEP, XL = L::XL, nl = L::nl, N1 = Fac<n>::N1, N2 = Fac<n>::N2;
  const int r0 = tile * XL, tid = thread_here(), lane = tid & 31, warp = tid >> 5;
  const size_t n3 = lv.n3, v0 = (size_t)r0 * n;
  float* f = reinterpret_cast<float*>(smem);
  if (J.precondition) {
    float2* sm = smem + tid % P;
    const int it0 = tid / P;
    const float* src = lv.tmp + v0;
#pragma unroll 1
    for (int r = warp; r < 3 * XL; r += X_WARPS) {
      const int c = r / XL, l = r - c * XL;
      line_load<n>(src + c * n3 + l * n, r0 + l < nl, lane, [&](int k, float x) { f[L::at(k, c, l)] = x; });
    }
    __syncthreads();
#pragma unroll 1
    for (int q = it0; q < n / 2 + 1; q += STEP) {
      const int nq = q ? n - q : 0;
      const float2 xq = sm[q * S], xn = q ? sm[nq * S] : make_float2(0.f, 0.f);
      float2 zq, zn;
      dct3_ends(xq, xn, __ldg(lv.tw4 + q), zq, zn);
      sm[q * S] = zq;
      if (q && 2 * q != n) sm[nq * S] = zn;
    }
    __syncthreads();
    inv_stage1<n, S, STEP>(sm, it0, lv.twm);
    __syncthreads();
    {
      float2 v[N2];
      inv_stage2<n, S>(v, sm, min(it0, N1 - 1));
      __syncthreads();  // the stage writes other rows than it reads
      if (it0 < N1) {
#pragma unroll
        for (int s = 0; s < N2; ++s) sm[esrc<n>(it0, s) * S] = v[s];
      }
    }
    __syncthreads();
  }
  if (J.ext_out) {  // pdg_precondition: the preconditioned gradient as [n^3][3], no update
    float* dst = J.ext_out + (size_t)r0 * n * 3;
#pragma unroll 1
    for (int l = warp; l < XL && r0 + l < nl; l += X_WARPS)
#pragma unroll 1
      for (int i = lane; i < 3 * n; i += 32) {
        const int e = i / 3, c = i - 3 * e;
        dst[(size_t)l * 3 * n + i] = f[L::at(e, c, l)];
      }
    return;
  }
  adam_tile<n>(J, lv, r0, tid, f);
}

// Items: the tiles of every line-path level of every job (three channels: the Cayley payload takes
// plane-path levels only).
template <bool FWD>
__global__ void __launch_bounds__(X_THREADS, 3) k_sob_x(const Plan* __restrict__ P) {
  extern __shared__ float2 smx[];
  __shared__ int2 zrange;
  const int nj = P->n_jobs;
  const int total = P->pre[ST_XTILE][nj];
  for (int it = blockIdx.x; it < total; it += gridDim.x) {
    const int j = find_job(P->pre[ST_XTILE], nj, it);
    const Job& J = *P->jobs[j];
    if (FWD && !J.precondition) continue;
    int t = it - P->pre[ST_XTILE][j];
    int l = J.L - 1, per = 0;
    for (; l >= 0; --l) {
      const int n = J.lev[l].n;
      if (!tile_level(n)) continue;
      per = x_tiles(n);
      if (t < per) break;
      t -= per;
    }
    if (l < 0) continue;
    const Level& lv = J.lev[l];
    __syncthreads();  // the previous item is done with the shared arrays
    if (FWD) {
      z_range(lv, &zrange);
      __syncthreads();
    }
    switch (lv.n) {
#define PDG_CASE(N)                           \
  case N:                                     \
    if (FWD) x_fwd<N>(J, lv, t, smx, zrange); \
    else x_inv<N>(J, lv, t, smx);             \
    break;
      PDG_LINE_SIZES(PDG_CASE)
#undef PDG_CASE
    }
  }
}

int x_smem_max(int nmax) {
  int m = 0;
  for (int n = 2; n <= nmax; ++n) m = std::max(m, x_smem(n));
  return m;
}

void sobolev_x_configure() {
  const int smem = x_smem_max(256);
  cudaFuncSetAttribute(k_sob_x<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  cudaFuncSetAttribute(k_sob_x<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

void launch_sobolev_x(const Plan* P, int grid, int nmax, bool fwd, cudaStream_t s) {
  const int smem = x_smem_max(nmax);
  if (fwd) k_sob_x<true><<<grid, X_THREADS, smem, s>>>(P);
  else k_sob_x<false><<<grid, X_THREADS, smem, s>>>(P);
}

}  // namespace pdg
