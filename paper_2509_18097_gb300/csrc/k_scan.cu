// Exclusive prefix sums used by the per-frame counting sorts: cell offsets of the point trees and
// row pointers of the per-level point -> vertex lists, over chunks of SCAN_CHUNK elements (chunk
// sums, a scan of the chunk sums, chunk scans).  All segments of a build share the three launches: a
// launch per level and array was a quarter of a frame's set-up.
#include "kernels.h"

namespace pdg {

// exclusive scan across a block of SCAN_THREADS (= 1024) threads; *total = block sum
template <class T>
__device__ __forceinline__ T block_excl_scan(T v, T* total) {
  __shared__ T ws[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  if (w == 0) {
    T t = ws[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    ws[lane] = t;
  }
  __syncthreads();
  const T pre = (w > 0 ? ws[w - 1] : 0) + x - v;
  if (total) *total = ws[31];
  __syncthreads();
  return pre;
}

__device__ __forceinline__ void load4(const int* in, int len, int base, int v[4]) {
  if (base + 3 < len) {
    const int4 q = *reinterpret_cast<const int4*>(in + base);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = (base + k < len) ? in[base + k] : 0;
  }
}

// exclusive scan of the chunk sums in place (one block); the total
template <class T>
__device__ T scan_sums(T* csum, int nch) {
  T carry = 0;
  for (int b = 0; b < nch; b += SCAN_THREADS) {
    const int i = b + threadIdx.x;
    const T v = i < nch ? csum[i] : 0;
    T tot;
    const T e = block_excl_scan(v, &tot);
    if (i < nch) csum[i] = carry + e;
    carry += tot;
  }
  return carry;
}

// ---- counts to offsets -------------------------------------------------------------------

struct ScanSegs {
  ScanSeg s[2];
  int pre[3];  // chunks before each segment
};

__global__ void __launch_bounds__(SCAN_THREADS) k_seg_scan_a(const ScanSegs g) {
  for (int it = blockIdx.x; it < g.pre[2]; it += gridDim.x) {
    const int k = it >= g.pre[1], chunk = it - g.pre[k];
    int v[4], tot;
    load4(g.s[k].in, g.s[k].len, chunk * SCAN_CHUNK + threadIdx.x * 4, v);
    block_excl_scan(v[0] + v[1] + v[2] + v[3], &tot);
    if (threadIdx.x == 0) g.s[k].csum[chunk] = tot;
  }
}
__global__ void __launch_bounds__(SCAN_THREADS) k_seg_scan_b(const ScanSegs g) {
  const ScanSeg& q = g.s[blockIdx.x];
  const int total = scan_sums(q.csum, g.pre[blockIdx.x + 1] - g.pre[blockIdx.x]);
  if (threadIdx.x == 0) q.out[q.len] = total;
}
__global__ void __launch_bounds__(SCAN_THREADS) k_seg_scan_c(const ScanSegs g) {
  for (int it = blockIdx.x; it < g.pre[2]; it += gridDim.x) {
    const int k = it >= g.pre[1], chunk = it - g.pre[k];
    const ScanSeg& q = g.s[k];
    const int base = chunk * SCAN_CHUNK + threadIdx.x * 4;
    int v[4];
    load4(q.in, q.len, base, v);
    int e = block_excl_scan(v[0] + v[1] + v[2] + v[3], (int*)nullptr) + q.csum[chunk];
    if (base + 3 < q.len) {
      int4 o;
      o.x = e; e += v[0];
      o.y = e; e += v[1];
      o.z = e; e += v[2];
      o.w = e;
      *reinterpret_cast<int4*>(q.out + base) = o;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (base + i < q.len) q.out[base + i] = e;
        e += v[i];
      }
    }
  }
}

void launch_scan(const ScanSeg& a, const ScanSeg& b, cudaStream_t s) {
  auto chunks = [](int len) { return (len + SCAN_CHUNK - 1) / SCAN_CHUNK; };
  const ScanSegs g{{a, b}, {0, chunks(a.len), chunks(a.len) + chunks(b.len)}};
  const int grid = std::max(1, std::min(g.pre[2], 2048));
  k_seg_scan_a<<<grid, SCAN_THREADS, 0, s>>>(g);
  k_seg_scan_b<<<2, SCAN_THREADS, 0, s>>>(g);
  k_seg_scan_c<<<grid, SCAN_THREADS, 0, s>>>(g);
}

// ---- interpolation lists -----------------------------------------------------------------
// Every level's per-vertex entry counts give its row pointers and, in the same scan, its active
// vertices (count > 0): a pair (entries, active vertices) in one 64-bit sum.

struct LevelChunks {
  int pre[MAXL + 1];  // chunks before each level
};

__device__ __forceinline__ int chunk_level(const LevelChunks& c, int L, int it) {
  int l = 0;
  while (l + 1 < L && it >= c.pre[l + 1]) ++l;
  return l;
}
__device__ __forceinline__ unsigned long long count_pair(int v) {
  return ((unsigned long long)(unsigned)v << 32) | (v > 0 ? 1u : 0u);
}

__global__ void __launch_bounds__(SCAN_THREADS) k_csr_scan_a(const Job* __restrict__ J, const LevelChunks c) {
  const int L = J->L;
  for (int it = blockIdx.x; it < c.pre[L]; it += gridDim.x) {
    const int l = chunk_level(c, L, it), chunk = it - c.pre[l];
    const Level& lv = J->lev[l];
    int v[4];
    load4(lv.cnt, lv.n3, chunk * SCAN_CHUNK + threadIdx.x * 4, v);
    unsigned long long tot;
    block_excl_scan(count_pair(v[0]) + count_pair(v[1]) + count_pair(v[2]) + count_pair(v[3]), &tot);
    if (threadIdx.x == 0) lv.csum[chunk] = tot;
  }
}

__global__ void __launch_bounds__(SCAN_THREADS) k_csr_scan_b(const Job* __restrict__ J, const LevelChunks c) {
  const int l = blockIdx.x;
  const Level& lv = J->lev[l];
  const unsigned long long total = scan_sums(lv.csum, c.pre[l + 1] - c.pre[l]);
  if (threadIdx.x == 0) {
    const int entries = (int)(total >> 32), active = (int)(total & 0xffffffffu);
    lv.rowptr[lv.n3] = entries;
    *lv.n_active = active;
    lv.act_ptr[active] = entries;
  }
}

// ... and marks the z-planes that hold an active vertex
__global__ void __launch_bounds__(SCAN_THREADS) k_csr_scan_c(const Job* __restrict__ J, const LevelChunks c) {
  const int L = J->L;
  for (int it = blockIdx.x; it < c.pre[L]; it += gridDim.x) {
    const int l = chunk_level(c, L, it), chunk = it - c.pre[l];
    const Level& lv = J->lev[l];
    const int base = chunk * SCAN_CHUNK + threadIdx.x * 4;
    int v[4];
    load4(lv.cnt, lv.n3, base, v);
    const unsigned long long e =
        block_excl_scan(count_pair(v[0]) + count_pair(v[1]) + count_pair(v[2]) + count_pair(v[3]),
                        (unsigned long long*)nullptr) +
        lv.csum[chunk];
    int row = (int)(e >> 32), act = (int)(e & 0xffffffffu), rows[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      rows[k] = row;
      if (v[k] > 0) {  // never past n3: load4 fills with 0
        lv.act_v[act] = base + k;
        lv.act_ptr[act] = row;
        lv.zmask[(base + k) / (lv.n * lv.n)] = 1;
        ++act;
      }
      row += v[k];
    }
    if (base + 3 < lv.n3) *reinterpret_cast<int4*>(lv.rowptr + base) = make_int4(rows[0], rows[1], rows[2], rows[3]);
    else
      for (int k = 0; k < 4 && base + k < lv.n3; ++k) lv.rowptr[base + k] = rows[k];
  }
}

void launch_csr_scan(const Job* J, const Job& hJ, cudaStream_t s) {
  LevelChunks c{};
  for (int l = 0; l < hJ.L; ++l) c.pre[l + 1] = c.pre[l] + (hJ.lev[l].n3 + SCAN_CHUNK - 1) / SCAN_CHUNK;
  const int grid = std::min(c.pre[hJ.L], 4096);
  k_csr_scan_a<<<grid, SCAN_THREADS, 0, s>>>(J, c);
  k_csr_scan_b<<<hJ.L, SCAN_THREADS, 0, s>>>(J, c);
  k_csr_scan_c<<<grid, SCAN_THREADS, 0, s>>>(J, c);
}

}  // namespace pdg
