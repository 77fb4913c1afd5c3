// y and z passes of the grid Sobolev preconditioner (Sec. 3.2, Eq. 3) by line transforms
// (sobolev_line.cuh): tiles of 2 P neighbouring lines of one channel.
//   y forward   DCT-II of the y-lines                                       tmp -> tmp
//   z           DCT-II, times (1 + lambda (mu_kx + mu_ky + mu_kz))^{-2} / n^3, inverse
//   y inverse
// L_l, the free-boundary 6-neighbour Laplacian, is the Kronecker sum of three path-graph
// Laplacians whose eigenvectors are the DCT-II basis vectors cos(pi k (i + 1/2) / n) with
// eigenvalues mu_k = 4 sin^2(pi k / 2n), so the operator is diagonal in that basis.
//
// What bounds them: at 256^3 a pass moves 403 MB (60 us at the copy rate) and takes 92 (y forward),
// 134 (z) and 121 us (y inverse), at 108^3 13 to 19 us; a warp-per-line Stockham FFT in shared memory
// took 484, 815 and 511 us.  Neither DRAM nor a pipe is full: a block's loads, stages and stores
// follow one another, so what counts is how many blocks overlap.  64 registers (4 blocks per SM; 92,
// 143, 122 us with the z pass of that time) beat 80 (98, 156, 134) and 48 (103, 150, 123).  Tiles of
// 32 line pairs at 32 <= n < 144 beat 16 (108^3: 13, 19, 13 against 15, 22, 15 us), whose stages fill
// half a block.
#include "sobolev_line.cuh"

namespace pdg {

constexpr int YZ_THREADS = 256;

template <int n, bool ZAXIS>
struct YZ {
  static constexpr int P = yz_pairs(n), nl = n * n, STRIDE = ZAXIS ? nl : n;
  static constexpr bool EVEN = n % 2 == 0;
  int a, b;              // the pair's lines (past nl: padding)
  float *ta, *tb;        // element 0 of each line
  bool ina, inb;

  // Even n: neighbouring lines, one float2 per element.  Odd n: lines P apart (a channel of n^3
  // floats and a row of n^2 are not 8-byte aligned there), two 4-byte accesses, each coalesced.
  __device__ __forceinline__ YZ(float* t, int r0, int p) {
    a = EVEN ? r0 + 2 * p : r0 + p;
    b = EVEN ? a + 1 : a + P;
    ina = a < nl;
    inb = b < nl;
    ta = t + (ZAXIS ? a : (a / n) * nl + a % n);
    tb = t + (ZAXIS ? b : (b / n) * nl + b % n);
  }
  __device__ __forceinline__ float2 load(int e) const {
    if (EVEN) return ina ? *reinterpret_cast<const float2*>(ta + e * STRIDE) : make_float2(0.f, 0.f);
    return make_float2(ina ? ta[e * STRIDE] : 0.f, inb ? tb[e * STRIDE] : 0.f);
  }
  __device__ __forceinline__ void store(int e, float2 v) const {
    if (EVEN) {
      if (ina) *reinterpret_cast<float2*>(ta + e * STRIDE) = v;
    } else {
      if (ina) ta[e * STRIDE] = v.x;
      if (inb) tb[e * STRIDE] = v.y;
    }
  }
};

// One tile in place in `t` (one channel of the level).  zr: the first z-plane with an active
// vertex and the number of planes up to the last one; the planes outside that range are zero and
// were not written by the passes before.
template <int n, int PASS>
__device__ __forceinline__ void yz_tile(const Level& lv, float* t, int tile, float2* smem, int2 zr) {
  using L = YZ<n, PASS == YZ_Z>;
  constexpr int P = L::P, N1 = Fac<n>::N1, N2 = Fac<n>::N2, nl = L::nl, STEP = YZ_THREADS / P;
  const int tid = thread_here(), p = tid % P, it0 = tid / P;
  const int r0 = tile * 2 * P;
  if (PASS == YZ_FWD)  // nothing to do when no plane of the tile is active
    if (min(r0 + 2 * P - 1, nl - 1) / n < zr.x || r0 / n >= zr.x + zr.y) return;
  L l(t, r0, p);
  float2* sm = smem + p;
  if (PASS != YZ_INV) {
    if (PASS == YZ_FWD) {
      l.ina = l.ina && (unsigned)(l.a / n - zr.x) < (unsigned)zr.y;
      l.inb = l.inb && (unsigned)(l.b / n - zr.x) < (unsigned)zr.y;
    }
#pragma unroll 1
    for (int s = it0; s < N1; s += STEP) {  // stage 1 straight from global memory
      float2 v[N2];
#pragma unroll
      for (int m = 0; m < N2; ++m) {
        const int e = esrc<n>(s, m);
        v[m] = PASS == YZ_FWD || (unsigned)(e - zr.x) < (unsigned)zr.y ? l.load(e) : make_float2(0.f, 0.f);
      }
      fwd_stage1<n, P>(v, sm, s, lv.twm);
    }
    __syncthreads();
    fwd_stage2<n, P, STEP>(sm, it0);
    __syncthreads();
  }
  // both ends of the spectrum together: separation and twiddle (forward), the spectral scale,
  // the inverse's input
  float ma = 0.f, mb = 0.f;
  if (PASS == YZ_Z) {  // the tile's lines are (kx, ky) columns, ky n + kx (padding wraps into range)
    ma = __ldg(lv.mu + l.a % n) + __ldg(lv.mu + l.a / n % n);
    mb = __ldg(lv.mu + l.b % n) + __ldg(lv.mu + l.b / n % n);
  }
  const float lam = lv.lam, inv_n3 = 1.f / ((float)n * n * n);
#pragma unroll 1
  for (int q = it0; q < n / 2 + 1; q += STEP) {
    const int nq = q ? n - q : 0;
    const bool two = q && 2 * q != n;  // q and n - q are different frequencies
    const float2 w = __ldg(lv.tw4 + q);
    float2 xq, xn;
    if (PASS == YZ_INV) {
      xq = l.load(q);
      xn = q ? l.load(nq) : make_float2(0.f, 0.f);
    } else {
      dct2_ends(sm[q * P], sm[nq * P], w, xq, xn);
    }
    if (PASS == YZ_FWD) {
      l.store(q, xq);
      if (two) l.store(nq, xn);
    } else {
      if (PASS == YZ_Z) {
        // A division per line: one shared by both, 1 / da = db / (da db), rounds more often, and its
        // products leave the range of float (NaN) long before 1 / da^2 does.  __fdividef (2 ulp) leaves
        // the preconditioner's error where an exact division has it (256^3: 3.12e-7 and 3.14e-7 RMS) and
        // the pass at 134 instead of 147 us; past 2^126 it gives 0, as the quotient nearly is.
        auto scale = [&](float m, float2 x) {
          const float da = fmaf(lam, ma + m, 1.f), db = fmaf(lam, mb + m, 1.f);
          return make_float2(x.x * __fdividef(inv_n3, da * da), x.y * __fdividef(inv_n3, db * db));
        };
        xq = scale(__ldg(lv.mu + q), xq);
        xn = q ? scale(__ldg(lv.mu + nq), xn) : make_float2(0.f, 0.f);
      }
      float2 zq, zn;
      dct3_ends(xq, xn, w, zq, zn);
      sm[q * P] = zq;
      if (two) sm[nq * P] = zn;
    }
  }
  if (PASS != YZ_FWD) {
    __syncthreads();
    inv_stage1<n, P, STEP>(sm, it0, lv.twm);
    __syncthreads();
#pragma unroll 1
    for (int k = it0; k < N1; k += STEP) {  // stage 2 straight to global memory
      float2 v[N2];
      inv_stage2<n, P>(v, sm, k);
#pragma unroll
      for (int s = 0; s < N2; ++s) l.store(esrc<n>(k, s), v[s]);
    }
  }
}

// Items: the tiles of every line-path level of every job, channel-major within a level.
template <int PASS>
__global__ void __launch_bounds__(YZ_THREADS, 4) k_sob_yz(const Plan* __restrict__ P) {
  extern __shared__ float2 smz[];
  __shared__ int2 zrange;
  const int nj = P->n_jobs;
  const int total = P->pre[ST_TILE][nj];
  for (int it = blockIdx.x; it < total; it += gridDim.x) {
    const int j = find_job(P->pre[ST_TILE], nj, it);
    const Job& J = *P->jobs[j];
    if (!J.precondition) continue;
    int t = it - P->pre[ST_TILE][j];
    int l = J.L - 1, per = 0;
    for (; l >= 0; --l) {
      const int n = J.lev[l].n;
      if (!tile_level(n)) continue;
      per = yz_tiles(n);
      if (t < J.C * per) break;
      t -= J.C * per;
    }
    if (l < 0) continue;
    const Level& lv = J.lev[l];
    const int c = t / per;
    const int tile = t - c * per;
    float* ch = lv.tmp + (size_t)c * lv.n3;
    __syncthreads();  // the previous item is done with the shared arrays
    if (PASS != YZ_INV) {
      z_range(lv, &zrange);
      __syncthreads();
    }
    switch (lv.n) {
#define PDG_CASE(N) \
  case N: yz_tile<N, PASS>(lv, ch, tile, smz, zrange); break;
      PDG_LINE_SIZES(PDG_CASE)
#undef PDG_CASE
    }
  }
}

int yz_smem_max(int nmax) {
  int m = 0;
  for (int n = 2; n <= nmax; ++n) m = std::max(m, n * yz_pairs(n) * (int)sizeof(float2));
  return m;
}

void sobolev_yz_configure() {
  const int smem = yz_smem_max(256);
  cudaFuncSetAttribute(k_sob_yz<YZ_FWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  cudaFuncSetAttribute(k_sob_yz<YZ_Z>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  cudaFuncSetAttribute(k_sob_yz<YZ_INV>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

void launch_sobolev_yz(const Plan* P, int grid, int nmax, int pass, cudaStream_t s) {
  const int smem = yz_smem_max(nmax);
  if (pass == YZ_FWD) k_sob_yz<YZ_FWD><<<grid, YZ_THREADS, smem, s>>>(P);
  else if (pass == YZ_Z) k_sob_yz<YZ_Z><<<grid, YZ_THREADS, smem, s>>>(P);
  else k_sob_yz<YZ_INV><<<grid, YZ_THREADS, smem, s>>>(P);
}

}  // namespace pdg
