// Internal device-side data structures and helpers shared by the kernels and the host
// runtime of libpdg (Preconditioned Deformation Grids, arXiv 2509.18097).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/pdg.h"

namespace pdg {

constexpr int MAXJ = 256;            // jobs (contexts) per batch
constexpr int MAXL = PDG_MAX_LEVELS; // grid levels
constexpr int SCAN_CHUNK = 4096;     // elements per scan chunk (1024 threads x 4)
constexpr int SCAN_THREADS = 1024;
constexpr int LEAF = 8;              // points per leaf of a point tree
constexpr int NODE = 32 * LEAF;      // points per node (32 leaves); 32 nodes make a super node
constexpr int LOSS_CHUNK = 2048;     // elements per loss-reduction chunk
constexpr double FX_SCALE = 1099511627776.0;  // 2^40: fixed-point scale of the reverse Chamfer sums

// A static-order box tree over the points of one or two sets, searched by k_nn.cu.  A set's points
// are sorted once per frame by the Hilbert index of their cell (`bits` per axis over the domain);
// slots of NODE consecutive points form a node, 32 nodes a super node, LEAF points a leaf.  A set
// starts on a node boundary, and its last node is padded with points at +infinity.  The order only
// decides how tight the boxes are: the search is exact for any order and any coordinates.
struct Tree {
  int bits;
  float lo[3];
  float inv_h[3];  // 2^bits / (hi - lo)
  int* hist;       // [sets 8^bits] per-cell counts; all zero between builds
  int* off;        // [sets 8^bits + 1] exclusive prefix of hist
  int* keys;       // [points] key of each point (scratch of the build)
  int* csum;       // scan chunk sums scratch
  int* perm;       // [slots] index of the slot's point, -1: padding
  float* pts;      // [leaves][3][LEAF] coordinates
  float4* lbox;    // [leaves][2] box of a leaf: (lo x, lo y, lo z, hi x), (hi y, hi z, -, -)
  float4* nbox;    // [nodes][2]
  float4* sbox;    // [super nodes][2], set 0 first
};

struct alignas(16) Level {  // 16: neighbouring fields in one load (k_deform, 1M points: 84.9 -> 81.6 us)
  int n;       // vertices per axis: 1 or 2^a 3^b
  int n3;      // n^3
  float sc_hi[3], sc_lo[3];  // (n - 1) / (hi - lo) per axis as a float pair (hi + lo)
  float lr;    // learning rate of the level (already x0.1 without preconditioning)
  float lam;   // lambda of the level
  float4* theta;  // [n3] values (x, y, z, 0): the displacement, or z of the Cayley payload
  float4* theta_t;  // [n3] translation t of the Cayley payload (null for the displacement payload)
  float* m;       // [C][n3] Adam first moment (channel-planar; C = 3, or 6: z then t)
  float* v;       // [C][n3] Adam second moment
  float* g;       // [C][n3] dLoss/dTheta (zero at vertices no point touches)
  float* tmp;     // [C][n3] spectral work array (and preconditioned gradient in debug mode)
  int* zmask;     // [n] 1 for z-planes that hold an active vertex (per frame); null: all planes
  float* piv;     // [(n/2 + 1) n^2] pivots of the z-direction twisted solves (n <= 128), per context
  int* piv_slow;  // device flag: some pivot past the first 16 differs from the limit (no register path)
  float* mu;      // [n] eigenvalues 4 sin^2(pi k / 2n) of the 1-D path Laplacian
  float2* tw;     // [n] FFT twiddles exp(-2 pi i k / n)
  float2* twm;    // [n] line path: twm[k N1 + t] = exp(-2 pi i t k / n) (N1 = line_n1(n))
  float2* tw4;    // [n] DCT twiddles exp(-i pi k / 2n)
  // point -> vertex interpolation lists, built once per frame (x is fixed in a frame)
  int* cnt;       // [n3] per-vertex entry counts (zero between builds)
  int* rowptr;    // [n3 + 1]
  int* act_v;     // [cap] active vertices (ascending)
  int* act_ptr;   // [cap + 1] entry range of each active vertex
  int2* ent;      // [8 Q] entries: (slot of the point, bits of the trilinear weight / L)
  int* n_active;  // device scalar
  unsigned long long* csum;  // scan scratch
  int adj_lg;     // adjoint: log2 of the lanes per row, 6 = a block per row (set by the plan kernel)
};

struct alignas(16) Job {
  int L;
  int C;                   // channels of the payload: 3 (displacement) or 6 (Cayley z, t)
  Level lev[MAXL];
  float lo[3], hi[3];
  float alpha, w_mesh, w_pts, w_iso;
  int stopgrad, precondition, keep_pgrad;
  float beta1, beta2, eps;
  int V, N, M, E, Q;       // template verts, source pts, target pts, edges, V + N
  int max_pts;
  float4* x;               // [Q] undeformed query points (template first), fixed in a frame
  float4* y;               // [Q] deformed points
  float4* gfwd;            // [Q] forward Chamfer gradient
  long long* acc;          // [Q][3] reverse Chamfer sums, fixed point (2^-40)
  float4* gy;              // [Q] dLoss/dy (= dLoss/dt with the Cayley payload)
  float4* gys;             // [slots of mov] the same in slot order, which the adjoint gathers from
  float4* zq;              // [Q] Cayley payload: the point's averaged z (null otherwise)
  float4* uq;              // [Q] Cayley payload: u = (I - Z)^{-1} x, so that R(z) x = 2 u - x
  float4* gz;              // [slots of mov] Cayley payload: dLoss/dz of the point, in slot order
  float* loss_fwd;         // [Q] phi(d^2) of each forward query
  float* loss_rev;         // [2 max_pts] phi(d^2) of each reverse query (set 0 then set 1)
  float* loss_iso;         // [E] |r_e|
  int* nn_fwd;             // [Q] (before the first search of a frame: its seed)
  int* nn_rev;             // [2 max_pts] (before the first search of a frame: its seed)
  float4* edge_d;          // [E] sgn(r) (y_i - y_j) / (|y_i - y_j| E)
  const int2* edges;       // [E]
  float* e_prev;           // [E] rest lengths from X_{t-1}
  const int* v2e_ptr;      // [V + 1]
  const int* v2e;          // [2E] (edge << 1) | (1 if the vertex is the edge's second end)
  float4* src4;            // [max_pts] current source cloud P_{t-1}
  float4* tgt4;            // [max_pts] target P_t
  float4* verts4;          // [V] current deformed template X_{t-1}
  Tree tgt;                // target points, built per frame
  Tree mov;                // two sets (template, source): order of the frame's x, boxes of the step's y
  int* slot_of;            // [Q] slot of a point
  float4* xs;              // [slots of mov] undeformed point and its index (bits) in slot order
  float* loss_part;        // [loss chunks][5] partial sums
  unsigned* gmax;          // max |dLoss/dy| component of the step (float bits; sets the adjoint's fixed-point scale)
  int* step;               // Adam step count k
  float* bias;             // [2] 1 / (1 - beta1^k), 1 / sqrt(1 - beta2^k) of the current step
  double* loss;            // [4] total, cd_mesh, cd_pts, iso of the last step
  int* status;             // sticky error flags (1: non-finite loss)
  unsigned long long* counters;  // [4] of the last step: NN candidates evaluated (counted only
                                 // when count_nn), NN queries decided by an exact tie,
                                 // 0, reserved
  const float* ext_in;     // pdg_precondition on a line-path level: the caller's gradient [n^3][3] ...
  float* ext_out;          // ... and where its preconditioned form goes (null in a step)
  int count_nn;            // 1: k_nn adds its candidate count to counters[0]
};

enum Counter { CNT_NN_CANDIDATES = 0, CNT_NN_TIES = 1 };

enum Stage { ST_Q = 0, ST_NODE, ST_SUPER, ST_NNF, ST_NNR, ST_E, ST_ADJ, ST_TILE, ST_ADJROW, ST_LOSSCH, ST_PLANE, ST_COL, ST_ADAM, ST_XTILE, NSTAGE };

struct Plan {
  int n_jobs;
  int pad_[3];
  Job* jobs[MAXJ];
  int pre[NSTAGE][MAXJ + 1];
};

// ------------------------------------------------------------------------------ helpers

// Which preconditioner path takes a level of n vertices per axis: powers of two up to 128
// (and n = 1) take the shared-memory plane path, 256 (whose plane does not fit) and the sizes with a
// factor 3 the line path.  Levels 16^3..128^3 together, with Adam: 125 us by planes, 177 us by lines.
__host__ __device__ __forceinline__ bool tile_level(int n) { return n > 128 || (n & (n - 1)) != 0; }

// Line path: sizes, line pairs of a y or z tile, x-lines (per channel) of an x tile.  A stage
// has about sqrt(n) work items per pair, so short lines go into larger tiles to fill a block.
#define PDG_LINE_SIZES(X)                                                                                    \
  X(3) X(6) X(9) X(12) X(18) X(24) X(27) X(36) X(48) X(54) X(72) X(81) X(96) X(108) X(144) X(162) X(192) \
  X(216) X(243) X(256)
// n = N1 x N2 with N1 <= N2, as even as the radices allow: the register DFTs of a line stay at
// 16 points or fewer, but for 162, 216 (18) and 243 (27)
__host__ __device__ constexpr int line_n1(int n) {
  return n <= 6      ? 1
         : n <= 12   ? 3
         : n == 18   ? 3
         : n == 24   ? 4
         : n == 27   ? 3
         : n <= 54   ? 6
         : n <= 72   ? 8
         : n == 81   ? 9
         : n == 96   ? 8
         : n == 108  ? 9
         : n == 144  ? 12
         : n == 162  ? 9
         : n <= 216  ? 12
         : n == 243  ? 9
                     : 16;
}
__host__ __device__ constexpr int yz_pairs(int n) { return n >= 144 ? 16 : n >= 32 ? 32 : 64; }
__host__ __device__ constexpr int x_lines(int n) { return n >= 64 ? 16 : n >= 24 ? 32 : 64; }
__host__ __device__ constexpr int yz_tiles(int n) { return (n * n + 2 * yz_pairs(n) - 1) / (2 * yz_pairs(n)); }
__host__ __device__ constexpr int x_tiles(int n) { return (n * n + x_lines(n) - 1) / x_lines(n); }

__device__ __forceinline__ int find_job(const int* pre, int n_jobs, int item) {
  int lo = 0, hi = n_jobs;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (__ldg(pre + mid) <= item) lo = mid; else hi = mid;
  }
  return lo;
}

// Sets of a tree as slot ranges.
struct SetRange {
  int slot0, n;    // first slot, points
  int node0, nodes;
  int super0, supers;
};
__host__ __device__ __forceinline__ SetRange set_range(int node0, int super0, int n) {
  SetRange r;
  r.slot0 = node0 * NODE;
  r.n = n;
  r.node0 = node0;
  r.nodes = (n + NODE - 1) / NODE;
  r.super0 = super0;
  r.supers = (r.nodes + 31) / 32;
  return r;
}
__device__ __forceinline__ SetRange mov_set(const Job& J, int set) {
  const SetRange a = set_range(0, 0, J.V);
  return set ? set_range(a.nodes, a.supers, J.N) : a;
}

__device__ __forceinline__ int cell_coord(float p, float lo, float inv_h, int G) {
  float t = (p - lo) * inv_h;
  t = fminf(fmaxf(t, -1.0f), (float)G);
  int c = (int)floorf(t);
  return min(max(c, 0), G - 1);
}

// Index of a cell along the Hilbert curve of 8^bits cells (the transposed-axes algorithm of
// Skilling, "Programming the Hilbert curve", 2004): unlike along the Morton curve, consecutive cells
// are neighbours, so 32 consecutive points rarely straddle distant parts of the surface.
__device__ __forceinline__ int hilbert3(int x, int y, int z, int bits) {
  int X[3] = {x, y, z};
  for (int q = 1 << (bits - 1); q > 1; q >>= 1) {
    const int p = q - 1;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (X[i] & q) {
        X[0] ^= p;
      } else {
        const int t = (X[0] ^ X[i]) & p;
        X[0] ^= t;
        X[i] ^= t;
      }
    }
  }
  X[1] ^= X[0];
  X[2] ^= X[1];
  int t = 0;
  for (int q = 1 << (bits - 1); q > 1; q >>= 1)
    if (X[2] & q) t ^= q - 1;
  int key = 0;
  for (int b = bits - 1; b >= 0; --b)
#pragma unroll
    for (int i = 0; i < 3; ++i) key = (key << 1) | (((X[i] ^ t) >> b) & 1);
  return key;
}

__device__ __forceinline__ int cell_key(const Tree& g, float x, float y, float z, int set) {
  const int G = 1 << g.bits;
  const int cx = cell_coord(x, g.lo[0], g.inv_h[0], G);
  const int cy = cell_coord(y, g.lo[1], g.inv_h[1], G);
  const int cz = cell_coord(z, g.lo[2], g.inv_h[2], G);
  return (set << (3 * g.bits)) + hilbert3(cx, cy, cz, g.bits);
}

// Stores the points of one node (thread t of 256: slot NODE nd + t; valid = false: padding) and
// the boxes of its leaves and of the node.  All 256 threads of the block; synchronises.
__device__ __forceinline__ void store_node(const Tree& T, int nd, float x, float y, float z, bool valid) {
  __shared__ float wbox[8][6];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const float inf = __int_as_float(0x7f800000);
  const int leaf = nd * (NODE / LEAF) + t / LEAF;
  float* p = T.pts + (size_t)leaf * (3 * LEAF) + (t & (LEAF - 1));
  p[0] = valid ? x : inf;
  p[LEAF] = valid ? y : inf;
  p[2 * LEAF] = valid ? z : inf;
  float b[6] = {valid ? x : inf, valid ? y : inf, valid ? z : inf, valid ? x : -inf, valid ? y : -inf, valid ? z : -inf};
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    if (o == LEAF && (lane & (LEAF - 1)) == 0) {
      T.lbox[2 * leaf] = make_float4(b[0], b[1], b[2], b[3]);
      T.lbox[2 * leaf + 1] = make_float4(b[4], b[5], 0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float v = __shfl_xor_sync(0xffffffffu, b[k], o);
      b[k] = k < 3 ? fminf(b[k], v) : fmaxf(b[k], v);
    }
  }
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < 6; ++k) wbox[warp][k] = b[k];
  __syncthreads();
  if (t == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w)
#pragma unroll
      for (int k = 0; k < 6; ++k) b[k] = k < 3 ? fminf(b[k], wbox[w][k]) : fmaxf(b[k], wbox[w][k]);
    T.nbox[2 * nd] = make_float4(b[0], b[1], b[2], b[3]);
    T.nbox[2 * nd + 1] = make_float4(b[4], b[5], 0.f, 0.f);
  }
  __syncthreads();
}

// squared distance, difference form; the same expression everywhere so that candidate
// comparisons are consistent between kernels
__device__ __forceinline__ float sqdist(float ax, float ay, float az, float bx, float by, float bz) {
  const float dx = __fsub_rn(ax, bx), dy = __fsub_rn(ay, by), dz = __fsub_rn(az, bz);
  return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}

// Grid coordinate of x in a level with n >= 2 vertices per axis (Eq. 1, vertex-aligned,
// clamped, last cell closed): u = (x - lo) (n - 1) / (hi - lo), i0 = min(floor(u), n - 2),
// f = u - i0.  x - lo is formed exactly (TwoSum) and multiplied by the scale held as a
// float pair with an FMA two-product, so f carries ~1 ulp of error instead of
// ulp(hi - lo) * (n - 1) (which would reach 1e-5 of a weight on 128^3 grids).
__device__ __forceinline__ void grid_coord(float x, float lo, float s_hi, float s_lo, int n, int& i0, float& f) {
  const float d = __fsub_rn(x, lo);
  const float bv = __fsub_rn(d, x);
  const float dl = __fadd_rn(__fsub_rn(x, __fsub_rn(d, bv)), __fsub_rn(-lo, bv));  // x - lo = d + dl exactly
  const float p = __fmul_rn(d, s_hi);
  const float e = __fmaf_rn(d, s_hi, -p);
  const float ul = __fadd_rn(e, __fmaf_rn(d, s_lo, __fmul_rn(dl, s_hi)));       // u = p + ul
  if (!(p > 0.f) && !(p == 0.f && ul > 0.f)) {  // u <= 0 (or NaN): clamp to vertex 0
    i0 = 0;
    f = 0.f;
    return;
  }
  if (p > (float)(n - 1) || (p == (float)(n - 1) && ul >= 0.f)) {  // u >= n - 1: clamp to the last vertex
    i0 = n - 2;
    f = 1.f;
    return;
  }
  float fl = floorf(p);
  if (fl == p && ul < 0.f) fl -= 1.f;
  int i = (int)fl;
  float fr = __fadd_rn(__fsub_rn(p, fl), ul);
  if (fr >= 1.f && i < n - 2) {
    i += 1;
    fr = __fsub_rn(fr, 1.f);
  }
  if (fr < 0.f && i > 0) {
    i -= 1;
    fr = __fadd_rn(fr, 1.f);
  }
  if (i > n - 2) {
    i = n - 2;
    fr = 1.f;
  }
  i0 = i;
  f = fminf(fmaxf(fr, 0.f), 1.f);
}

// The Cayley rotation of Sec. 3.3 applied to x without forming R(z) = (I + Z)(I - Z)^{-1}:
// (I - Z)^{-1} = (I + Z + z z^T) / (1 + |z|^2) (multiply out with Z^2 = z z^T - |z|^2 I), and
// R = 2 (I - Z)^{-1} - I, so R(z) x = 2 u - x with u = (x + z x x + z (z . x)) / (1 + |z|^2).
__device__ __forceinline__ float3 cross3(float3 a, float3 b) {
  return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}

__device__ __forceinline__ float3 cayley_u(float3 z, float3 x) {
  const float s = 1.f / (1.f + (z.x * z.x + z.y * z.y + z.z * z.z));
  const float zx = z.x * x.x + z.y * x.y + z.z * x.z;
  const float3 c = cross3(z, x);
  return make_float3((x.x + c.x + z.x * zx) * s, (x.y + c.y + z.y * zx) * s, (x.z + c.z + z.z * zx) * s);
}

// dLoss/dz for y = R(z) x + t and g = dLoss/dy: d(R x) = 2 (I - Z)^{-1} dZ u = -2 (I - Z)^{-1} [u]x dz,
// so dLoss/dz = 2 u x w with w = (I - Z)^{-T} g = (I + Z)^{-1} g = (g - z x g + z (z . g)) / (1 + |z|^2).
__device__ __forceinline__ float3 cayley_grad_z(float3 z, float3 u, float3 g) {
  const float s = 1.f / (1.f + (z.x * z.x + z.y * z.y + z.z * z.z));
  const float zg = z.x * g.x + z.y * g.y + z.z * g.z;
  const float3 c = cross3(z, g);
  const float3 w = make_float3((g.x - c.x + z.x * zg) * s, (g.y - c.y + z.y * zg) * s, (g.z - c.z + z.z * zg) * s);
  const float3 r = cross3(u, w);
  return make_float3(2.f * r.x, 2.f * r.y, 2.f * r.z);
}

__device__ __forceinline__ long long to_fx(float v) { return __float2ll_rn(v * 1099511627776.0f); }
__device__ __forceinline__ float from_fx(long long a) { return __ll2float_rn(a) * (1.0f / 1099511627776.0f); }

}  // namespace pdg
