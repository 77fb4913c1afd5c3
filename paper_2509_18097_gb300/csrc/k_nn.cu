// Exact nearest neighbours for the bidirectional robust Chamfer distance (Sec. 3.4) and
// its gradient.  Four searches per step: template vertices and source points (the moving
// sets) against the target cloud, and the target cloud against each moving set.
//
// A warp takes 32 / SUB neighbouring queries (consecutive slots of their own tree), SUB lanes each,
// through the box tree of the searched set together (see Tree).  At the upper levels the 32 lanes
// test 32 boxes against the box of the warp's queries: a box farther away than the worst of the
// warp's best distances holds nothing for any query.  The leaves that survive are listed; each
// sub-lane of a query takes every SUB-th of them, tests it against its own query and best distance,
// and evaluates its 8 points (two points per packed FP32 instruction).  Queries start from their
// neighbour of the previous step, a point of the set, so the bounds are tight from the first box on.
//
// Why this split.  About 8 leaves per query pass its own bound (100k points, neighbours 4 spacings
// away), 26 that of any of 32 neighbouring queries: a warp of 32 queries evaluates 3 times what one
// query needs, and its chain of dependent box loads (about 20 us whatever the size) leaves a small
// problem waiting.  Fewer queries per warp shorten both and repeat the upper levels.  Step times,
// SUB = 1 / 2 / 4 / 8: 100k points 275 / 268 / 272 / 307 us, 20k (Cayley) 288 / 278 / 280 / 285,
// 2k 66 / 62 / 58 / 57; so SUB = 8 below 4 warps of 32 queries per SM and 2 above.
// What bounds it: register write-back of L1 loads (a leaf is 96 bytes to every lane) and latency,
// 0.5 instructions per cycle and scheduler.  It replaces a thread per query over 3x3x3 boxes of
// 32-point cells with the moving points re-sorted each step: at 100k points (searches, sort, ring
// pass) 157 us of launches; the order of the points is now the frame's, and only boxes are redone.
//
// Exactness: candidates are compared with one fp32 expression (sqdist).  The bounds use the same
// operations in the same order on differences that rounding cannot carry past the true ones
// (subtraction, product and fused sum are monotone in fp32), so a box's bound never exceeds the
// fp32 squared distance of a point in it, and only strictly larger bounds are skipped.  The result
// is the exact lexicographic minimum of (fp32 d^2, index) over the whole set.
#include <float.h>

#include "kernels.h"

namespace pdg {

constexpr int NN_THREADS = 128;

// ------------------------------------------------------------------------------ finalise

struct QueryRef {
  float x, y, z;
  int id;    // Q index (forward) or target index (reverse), -1: padding
  int set;   // moving set searched (reverse)
};

// The loss term phi(s) = s e^{-alpha s} and the gradient 2 phi'(s) (a - b) of a matched
// pair (Sec. 3.4); phi'(s) = e^{-alpha s}(1 - alpha s), or e^{-alpha s} with the stop-gradient.
// d2, idx: the nearest point (idx < 0: none found, non-finite coordinates).
template <bool FWD>
__device__ __forceinline__ void finalize(const Job& J, const QueryRef& q, float d2, int idx) {
  if (idx < 0) {
    if (FWD) {
      J.loss_fwd[q.id] = __int_as_float(0x7fc00000);
      J.gfwd[q.id] = make_float4(0.f, 0.f, 0.f, 0.f);
      J.nn_fwd[q.id] = -1;
    } else {
      J.loss_rev[q.set * J.M + q.id] = __int_as_float(0x7fc00000);
      J.nn_rev[q.set * J.M + q.id] = -1;
    }
    return;
  }
  const float s = d2;
  const float e = expf(-J.alpha * s);
  const float phi = s * e;
  const float dphi = J.stopgrad ? e : e * (1.f - J.alpha * s);
  if (FWD) {  // moving point a = q -> target point b
    const float4 t = J.tgt4[idx];
    const bool mesh = q.id < J.V;
    const float coef = 2.f * dphi * (mesh ? J.w_mesh / (float)J.V : J.w_pts / (float)(J.Q - J.V));
    J.loss_fwd[q.id] = phi;
    J.gfwd[q.id] = make_float4(coef * (q.x - t.x), coef * (q.y - t.y), coef * (q.z - t.z), 0.f);
    J.nn_fwd[q.id] = idx;
  } else {  // target point q -> moving point a of set q.set; the gradient goes to a
    const float4 a = J.y[idx];
    J.loss_rev[q.set * J.M + q.id] = phi;
    J.nn_rev[q.set * J.M + q.id] = idx - (q.set ? J.V : 0);
    const float c = 2.f * dphi;
    unsigned long long* acc = reinterpret_cast<unsigned long long*>(J.acc + 3 * (size_t)idx);
    atomicAdd(acc + 0, (unsigned long long)to_fx(c * (a.x - q.x)));
    atomicAdd(acc + 1, (unsigned long long)to_fx(c * (a.y - q.y)));
    atomicAdd(acc + 2, (unsigned long long)to_fx(c * (a.z - q.z)));
  }
}

// ------------------------------------------------------------------------------ bounds

struct Box {
  float4 a;  // lo x, lo y, lo z, hi x
  float2 c;  // hi y, hi z
};

__device__ __forceinline__ Box load_box(const float4* b, int i) {
  Box r;
  r.a = __ldg(b + 2 * i);
  r.c = __ldg(reinterpret_cast<const float2*>(b + 2 * i + 1));
  return r;
}

// fp32 lower bound on sqdist between any point in [l, h] and any point of the box
__device__ __forceinline__ float box_lb(const Box& b, float lx, float ly, float lz, float hx, float hy, float hz) {
  const float dx = fmaxf(fmaxf(__fsub_rn(b.a.x, hx), __fsub_rn(lx, b.a.w)), 0.f);
  const float dy = fmaxf(fmaxf(__fsub_rn(b.a.y, hy), __fsub_rn(ly, b.c.x)), 0.f);
  const float dz = fmaxf(fmaxf(__fsub_rn(b.a.z, hz), __fsub_rn(lz, b.c.y)), 0.f);
  return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}

// minimum / maximum over the warp (signed floats as order-preserving integers)
__device__ __forceinline__ int ord(float f) {
  const int i = __float_as_int(f);
  return i < 0 ? i ^ 0x7fffffff : i;
}
__device__ __forceinline__ float warp_min(float f) {
  const int m = __reduce_min_sync(0xffffffffu, ord(f));
  return __int_as_float(m < 0 ? m ^ 0x7fffffff : m);
}
__device__ __forceinline__ float warp_max(float f) {
  const int m = __reduce_max_sync(0xffffffffu, ord(f));
  return __int_as_float(m < 0 ? m ^ 0x7fffffff : m);
}

// ------------------------------------------------------------------------------ leaves

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Squared distances to the 8 points of a leaf, bitwise sqdist (its differences only change sign)
struct NegQuery {
  f32x2 x, y, z;  // (-q, -q) per axis
};
__device__ __forceinline__ void leaf_d2(const float* pts, int leaf, const NegQuery& q, float (&d)[LEAF]) {
  const ulonglong2* p = reinterpret_cast<const ulonglong2*>(pts + (size_t)leaf * (3 * LEAF));
  const ulonglong2 xa = __ldg(p), xb = __ldg(p + 1), ya = __ldg(p + 2), yb = __ldg(p + 3), za = __ldg(p + 4),
                   zb = __ldg(p + 5);
  const f32x2 x[4] = {xa.x, xa.y, xb.x, xb.y}, y[4] = {ya.x, ya.y, yb.x, yb.y}, z[4] = {za.x, za.y, zb.x, zb.y};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const f32x2 dx = add2(x[k], q.x), dy = add2(y[k], q.y), dz = add2(z[k], q.z);
    const float2 s = unpack2(fma2(dz, dz, fma2(dy, dy, mul2(dx, dx))));
    d[2 * k] = s.x;
    d[2 * k + 1] = s.y;
  }
}

// lowest index among a leaf's points at squared distance d2 (and how many there are)
__device__ __forceinline__ int leaf_index(const Tree& T, int leaf, const NegQuery& q, float d2, int& count) {
  float d[LEAF];
  leaf_d2(T.pts, leaf, q, d);
  int id = 0x7fffffff;
  count = 0;
#pragma unroll
  for (int k = 0; k < LEAF; ++k)
    if (d[k] == d2) {
      id = min(id, __ldg(T.perm + leaf * LEAF + k));
      ++count;
    }
  return id;
}

// Best so far of a lane: d2, and the leaf that holds a point at that distance (-1: none yet).
// tie: another leaf holds an equally near point.
struct Best {
  float d2;
  int leaf;
  bool tie;
};

__device__ __forceinline__ void eval_leaf(const Tree& T, int leaf, const NegQuery& q, Best& b) {
  float d[LEAF];
  leaf_d2(T.pts, leaf, q, d);
  const float m = fminf(fminf(fminf(d[0], d[1]), fminf(d[2], d[3])), fminf(fminf(d[4], d[5]), fminf(d[6], d[7])));
  if (m < b.d2) {
    b.d2 = m;
    b.leaf = leaf;
    b.tie = false;
  } else if (m == b.d2 && b.leaf >= 0 && leaf != b.leaf) {  // an exact tie: keep the leaf with the lower index
    int c;
    if (leaf_index(T, leaf, q, m, c) < leaf_index(T, b.leaf, q, m, c)) b.leaf = leaf;
    b.tie = true;
  }
}

// ------------------------------------------------------------------------------ search

struct WarpBox {
  float lx, ly, lz, hx, hy, hz;
};

// A warp's traversal.  SUB lanes share a query (lane = sub (32 / SUB) + query): each takes other leaves,
// and their results are merged at the end.
template <int SUB, bool COUNT>
struct Search {
  static constexpr int QPW = 32 / SUB, LIST = 64;
  const Tree& T;
  QueryRef q;
  NegQuery nq;
  WarpBox w;
  Best b;
  float lim;   // no worse than the best distance of the query's lanes: what is farther is skipped
  float wmax;  // largest lim of the warp
  int* list;   // the warp's list of leaves to look at
  int n;
  int nc;      // candidates evaluated by this lane (counting instance)

  __device__ __forceinline__ void update_limits() {
    lim = fminf(lim, b.d2);
#pragma unroll
    for (int o = QPW; o < 32; o <<= 1) lim = fminf(lim, __shfl_xor_sync(0xffffffffu, lim, o));
    wmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(lim, 0.f))));
  }

  __device__ __forceinline__ bool wanted(int leaf) const {
    return box_lb(load_box(T.lbox, leaf), q.x, q.y, q.z, q.x, q.y, q.z) <= lim;
  }

  // looks at the listed leaves, one per sub-lane at a time
  __device__ __forceinline__ void flush() {
    __syncwarp();
#pragma unroll 1
    for (int i = 0; i < n; i += SUB) {
      const int k = i + threadIdx.x % 32 / QPW;
      const int leaf = list[min(k, n - 1)];
      if (k < n && wanted(leaf)) {
        eval_leaf(T, leaf, nq, b);
        lim = fminf(lim, b.d2);
        if (COUNT) nc += LEAF;
      }
    }
    __syncwarp();
    n = 0;
    update_limits();
  }

  // lists the leaves of a node that the warp's box may need
  __device__ __forceinline__ void node(int nd) {
    const int lane = threadIdx.x & 31;
    const bool in = box_lb(load_box(T.lbox, nd * 32 + lane), w.lx, w.ly, w.lz, w.hx, w.hy, w.hz) <= wmax;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (in) list[n + __popc(m & ((1u << lane) - 1u))] = nd * 32 + lane;
    n += __popc(m);
    if (n > LIST - 32) flush();
  }
};

// items: SUB warps for each 32 queries (ST_NNF: moving slots, template set first; ST_NNR: target
// slots, searched in the tree of the moving set `set`)
template <bool FWD, int SUB, bool COUNT>
__global__ void __launch_bounds__(NN_THREADS, 8) k_nn(const Plan* __restrict__ P, int set) {
  constexpr int ST = FWD ? ST_NNF : ST_NNR, QPW = 32 / SUB;
  __shared__ int lists[NN_THREADS / 32][Search<SUB, COUNT>::LIST];
  const int nj = P->n_jobs;
  const int total = P->pre[ST][nj] * SUB;
  const int lane = threadIdx.x & 31;
  for (int it = (blockIdx.x * NN_THREADS + threadIdx.x) >> 5; it < total; it += gridDim.x * (NN_THREADS / 32)) {
    const int j = find_job(P->pre[ST], nj, it / SUB);
    const Job& J = *P->jobs[j];
    const int t = it / SUB - P->pre[ST][j];
    const Tree& own = FWD ? J.mov : J.tgt;
    Search<SUB, COUNT> s{FWD ? J.tgt : J.mov};
    QueryRef& q = s.q;
    q.set = FWD ? 0 : set;
    int slot = 32 * t + it % SUB * QPW + lane % QPW;
    if (FWD) {
      const int w0 = (J.V + 31) / 32;
      if (t >= w0) slot += mov_set(J, 1).slot0 - 32 * w0;
    }
    const SetRange r = FWD ? set_range(0, 0, J.M) : mov_set(J, q.set);
    const float* p = own.pts + (size_t)(slot / LEAF) * (3 * LEAF) + slot % LEAF;
    q.id = own.perm[slot];
    q.x = p[0];
    q.y = p[LEAF];
    q.z = p[2 * LEAF];
    // a query with a NaN coordinate has no nearest point; like a padding lane it asks for nothing
    const bool live = q.id >= 0 && q.x == q.x && q.y == q.y && q.z == q.z;
    s.b = Best{live ? FLT_MAX : -1.f, -1, false};
    if (live) {
      // Warm start: the distance of the previous step's neighbour (k_nn_seed's point in a frame's first
      // step) at its current position, one ulp up, so that its own leaf counts as an improvement and
      // records itself.
      const int w = FWD ? J.nn_fwd[q.id] : J.nn_rev[q.set * J.M + q.id];
      if (w >= 0) {
        const float4 c = FWD ? J.tgt4[w] : J.y[w + (q.set ? J.V : 0)];
        const float d2 = sqdist(q.x, q.y, q.z, c.x, c.y, c.z);
        if (d2 < FLT_MAX) s.b.d2 = __uint_as_float(__float_as_uint(d2) + 1u);
      }
    }
    s.nq = NegQuery{pack2(-q.x, -q.x), pack2(-q.y, -q.y), pack2(-q.z, -q.z)};
    const float inf = __int_as_float(0x7f800000);
    WarpBox& w = s.w;
    w.lx = warp_min(live ? q.x : inf);
    w.ly = warp_min(live ? q.y : inf);
    w.lz = warp_min(live ? q.z : inf);
    w.hx = warp_max(live ? q.x : -inf);
    w.hy = warp_max(live ? q.y : -inf);
    w.hz = warp_max(live ? q.z : -inf);
    s.list = lists[threadIdx.x >> 5];
    s.n = s.nc = 0;
    s.lim = s.b.d2;
    s.update_limits();
    if (__any_sync(0xffffffffu, live)) {
      for (int s0 = 0; s0 < r.supers; s0 += 32) {
        float lbs = inf;
        if (s0 + lane < r.supers)
          lbs = box_lb(load_box(s.T.sbox, r.super0 + s0 + lane), w.lx, w.ly, w.lz, w.hx, w.hy, w.hz);
        unsigned ms = __ballot_sync(0xffffffffu, lbs <= s.wmax);
        while (ms) {
          const int sn = s0 + __ffs(ms) - 1;
          ms &= ms - 1;
          float lbn = inf;
          if (32 * sn + lane < r.nodes)
            lbn = box_lb(load_box(s.T.nbox, r.node0 + 32 * sn + lane), w.lx, w.ly, w.lz, w.hx, w.hy, w.hz);
          unsigned mn = __ballot_sync(0xffffffffu, lbn <= s.wmax);
          while (mn) {
            const int nd = r.node0 + 32 * sn + __ffs(mn) - 1;
            mn &= mn - 1;
            // the warp's box can be much larger than its queries (a jump of the curve): ask the lanes
            const Box box = load_box(s.T.nbox, nd);
            if (__any_sync(0xffffffffu, box_lb(box, q.x, q.y, q.z, q.x, q.y, q.z) <= s.lim)) s.node(nd);
          }
        }
      }
      if (s.n) s.flush();
    }
    if (COUNT) {
      const unsigned c = __reduce_add_sync(0xffffffffu, q.id >= 0 ? (unsigned)s.nc : 0u);
      if (lane == 0) atomicAdd(J.counters + CNT_NN_CANDIDATES, (unsigned long long)c);
    }
    int idx = -1;
    bool tie = s.b.tie;
    if (s.b.leaf >= 0) {
      int count;
      idx = leaf_index(s.T, s.b.leaf, s.nq, s.b.d2, count);
      tie = tie || count > 1;
    }
    float d2 = idx >= 0 ? s.b.d2 : inf;
#pragma unroll
    for (int o = QPW; o < 32; o <<= 1) {  // the lexicographic minimum over the query's lanes
      const float d = __shfl_xor_sync(0xffffffffu, d2, o);
      const int i = __shfl_xor_sync(0xffffffffu, idx, o);
      const bool ti = __shfl_xor_sync(0xffffffffu, tie, o);
      if (i >= 0 && (d < d2 || idx < 0)) {
        d2 = d;
        idx = i;
        tie = ti;
      } else if (i >= 0 && d == d2) {
        tie = tie || ti || i != idx;
        idx = min(idx, i);
      }
    }
    if (q.id >= 0 && lane < QPW) {
      if (COUNT && idx >= 0 && tie) atomicAdd(J.counters + CNT_NN_TIES, 1ull);
      finalize<FWD>(J, q, d2, idx);
    }
    __syncwarp();
  }
}

// A frame's first neighbours: a point of the query's own cell of the searched set's sort, or the next
// one along the curve where that cell is empty.  Any point of the set will do; without one the first
// step's searches would start from no bound (first evaluation at 100k points: about 100 us more).
__global__ void k_nn_seed(Job* __restrict__ Jp) {
  const Job& J = *Jp;
  const int total = J.Q + (J.N > 0 ? 2 : 1) * J.M;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    if (i < J.Q) {
      const float4 x = J.x[i];
      J.nn_fwd[i] = J.tgt.perm[min(J.tgt.off[cell_key(J.tgt, x.x, x.y, x.z, 0)], J.M - 1)];
    } else {
      const int set = i - J.Q >= J.M, t = i - J.Q - set * J.M;
      const float4 x = J.tgt4[t];
      const SetRange r = mov_set(J, set);
      const int pos = J.mov.off[cell_key(J.mov, x.x, x.y, x.z, set)] - (set ? J.V : 0);
      J.nn_rev[i - J.Q] = J.mov.perm[r.slot0 + min(pos, r.n - 1)] - (set ? J.V : 0);
    }
  }
}

void launch_nn_seed(Job* J, const Job& hJ, cudaStream_t s) {
  const int n = hJ.Q + 2 * hJ.M;
  k_nn_seed<<<std::min((n + 255) / 256, 4096), 256, 0, s>>>(J);
}

template <int SUB>
static void launch_nn_sub(const Plan* P, int grid, cudaStream_t s, int set, bool count) {
  if (set < 0 && count) k_nn<true, SUB, true><<<grid, NN_THREADS, 0, s>>>(P, 0);
  else if (set < 0) k_nn<true, SUB, false><<<grid, NN_THREADS, 0, s>>>(P, 0);
  else if (count) k_nn<false, SUB, true><<<grid, NN_THREADS, 0, s>>>(P, set);
  else k_nn<false, SUB, false><<<grid, NN_THREADS, 0, s>>>(P, set);
}

void launch_nn(const Plan* P, int grid, cudaStream_t s, int set, int sub, bool count) {
  if (sub == 2) launch_nn_sub<2>(P, grid, s, set, count);
  else launch_nn_sub<8>(P, grid, s, set, count);
}

}  // namespace pdg
