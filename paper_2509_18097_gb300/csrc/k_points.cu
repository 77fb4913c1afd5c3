// Point- and edge-parallel kernels of the step: the plan, multi-level trilinear
// evaluation (Eq. 1), the boxes of the moving trees, edge isometry (Sec. 3.4), gradient
// assembly and the loss reduction; plus the per-frame set-up kernels.
#include "kernels.h"

namespace pdg {

// ------------------------------------------------------------------------------ plan

// Start of a step for one job, done by the thread of the job's first point in k_interp.
// bump = 1: a new optimisation step (advances the Adam step count and its bias corrections
// and clears the per-step counters); bump = 2: an evaluation (clears the counters only).
__device__ __forceinline__ void job_bump(const Job& J, int bump) {
  *J.gmax = 0u;
  J.counters[CNT_NN_CANDIDATES] = 0ull;
  J.counters[CNT_NN_TIES] = 0ull;
  if (bump == 1) {
    const int k = *J.step + 1;
    *J.step = k;
    // 1 - beta^k = -expm1(k log1p(beta - 1)): no cancellation for small k (beta - 1 is exact)
    J.bias[0] = 1.f / -expm1f((float)k * log1pf(J.beta1 - 1.f));
    J.bias[1] = rsqrtf(-expm1f((float)k * log1pf(J.beta2 - 1.f)));
  }
}

// Computes, on the device, the per-stage item prefixes over the jobs of a plan.  They change
// only when a job starts a frame (its active-vertex counts) or the membership changes, so
// the host launches this outside the per-step graph, when the plan is stale.  One block.
__global__ void k_plan(Plan* P) {
  __shared__ int cnt[NSTAGE][MAXJ];
  const int nj = P->n_jobs;
  for (int j = threadIdx.x; j < nj; j += blockDim.x) {
    Job* J = P->jobs[j];
    cnt[ST_Q][j] = J->Q;
    // reverse queries into the source set only when there is one (a template-mesh fit has none)
    const int nrs = J->N > 0 ? 2 : 1;
    const SetRange s0 = mov_set(*J, 0), s1 = mov_set(*J, 1);
    cnt[ST_NODE][j] = s0.nodes + s1.nodes;
    cnt[ST_SUPER][j] = s0.supers + s1.supers;
    cnt[ST_NNF][j] = (J->V + 31) / 32 + (J->N + 31) / 32;  // warps of 32 queries
    cnt[ST_NNR][j] = (J->M + 31) / 32;  // per moving set
    cnt[ST_E][j] = J->E;
    int a = 0, t = 0, xt = 0, p3 = 0, cols = 0, ad = 0;
    int aw = 0;
    // the levels' loads are independent: issue them level-parallel (a dependent chain of
    // global loads per level would put a dozen memory latencies on the step's critical path)
    const int L = J->L;
    int na_l[MAXL], ne_l[MAXL];
#pragma unroll
    for (int l = 0; l < MAXL; ++l) na_l[l] = l < L ? *J->lev[l].n_active : 0;
#pragma unroll
    for (int l = 0; l < MAXL; ++l) ne_l[l] = na_l[l] > 0 ? J->lev[l].act_ptr[na_l[l]] : 0;
#pragma unroll
    for (int l = 0; l < MAXL; ++l) {
      if (l >= L) break;
      // adjoint: 2^adj_lg lanes per row, 8 to 16 entries per lane
      // (a row holds one entry per point in the 8 cells around its vertex: a few dozen on
      // fine levels, thousands on coarse ones), so a warp sums 32 >> adj_lg rows; rows of
      // 512 entries or more on average (adj_lg = 6) get a whole block each
      Level& lv = J->lev[l];
      const int na = na_l[l];
      const int ne = ne_l[l];
      const int avg = ne / max(na, 1);
      int lg = 0;
      while (lg < 6 && (16 << lg) <= avg) ++lg;
      lv.adj_lg = lg;
      if (lg == 6) a += na;
      else aw += (na + (32 >> lg) - 1) >> (5 - lg);
      if (tile_level(J->lev[l].n)) {
        t += J->C * yz_tiles(J->lev[l].n);
        xt += x_tiles(J->lev[l].n);
      } else {
        p3 += J->lev[l].n;
        cols += J->C * ((J->lev[l].n * J->lev[l].n + 63) / 64);  // blocks of 64 columns (two threads each)
        ad += (J->lev[l].n3 + 3) >> 2;
      }
    }
    cnt[ST_ADJROW][j] = a;
    cnt[ST_ADJ][j] = aw;
    cnt[ST_TILE][j] = t;
    cnt[ST_XTILE][j] = xt;
    cnt[ST_PLANE][j] = J->C * p3;
    cnt[ST_COL][j] = cols;
    cnt[ST_ADAM][j] = ad;
    cnt[ST_LOSSCH][j] = (J->Q + nrs * J->M + J->E + LOSS_CHUNK - 1) / LOSS_CHUNK;
  }
  __syncthreads();
  if (threadIdx.x < NSTAGE) {
    const int s = threadIdx.x;
    int acc = 0;
    P->pre[s][0] = 0;
    for (int j = 0; j < nj; ++j) {
      acc += cnt[s][j];
      P->pre[s][j + 1] = acc;
    }
  }
}

// the job record (by value, in the launch's arguments) and, if given, the plan that holds it alone
__global__ void k_op_job(const __grid_constant__ Job job, Job* dJ, Plan* dP) {
  const unsigned* src = reinterpret_cast<const unsigned*>(&job);
  unsigned* dst = reinterpret_cast<unsigned*>(dJ);
  for (int i = threadIdx.x; i < (int)(sizeof(Job) / 4); i += blockDim.x) dst[i] = src[i];
  if (dP && threadIdx.x == 0) {
    dP->n_jobs = 1;
    dP->jobs[0] = dJ;
  }
}

// ------------------------------------------------------------------------------ (a) eval

// Trilinear interpolation of one level's values at a point (Eq. 1; vertex-aligned levels,
// coordinates clamped to the domain, last cell closed): the cell's first vertex and the
// fractional coordinates, computed once and used for each payload array of the level.  A
// level of one vertex has the constant value v[0].
struct LevelCoord {
  int base;  // flat index of the cell's (0, 0, 0) corner
  int n;
  float fx, fy, fz;
};

__device__ __forceinline__ LevelCoord level_coord(const Job& J, const Level& lv, float px, float py, float pz) {
  LevelCoord c;
  c.n = lv.n;
  if (lv.n == 1) {
    c.base = 0;
    c.fx = c.fy = c.fz = 0.f;
    return c;
  }
  int ix, iy, iz;
  grid_coord(px, J.lo[0], lv.sc_hi[0], lv.sc_lo[0], lv.n, ix, c.fx);
  grid_coord(py, J.lo[1], lv.sc_hi[1], lv.sc_lo[1], lv.n, iy, c.fy);
  grid_coord(pz, J.lo[2], lv.sc_hi[2], lv.sc_lo[2], lv.n, iz, c.fz);
  c.base = (iz * lv.n + iy) * lv.n + ix;
  return c;
}

// adds sum_corners w * v[corner] to u (all 8 corner loads issued before any is used)
__device__ __forceinline__ void level_add(const LevelCoord& L, const float4* __restrict__ v, float& ux, float& uy,
                                          float& uz) {
  if (L.n == 1) {
    const float4 c = v[0];
    ux += c.x; uy += c.y; uz += c.z;
    return;
  }
  const int n = L.n;
  const float4* t0 = v + L.base;
  const float4* t1 = t0 + (size_t)n * n;
  const float4 c000 = t0[0], c100 = t0[1], c010 = t0[n], c110 = t0[n + 1];
  const float4 c001 = t1[0], c101 = t1[1], c011 = t1[n], c111 = t1[n + 1];
  const float fx = L.fx, fy = L.fy, fz = L.fz;
  const float gx = 1.f - fx, gy = 1.f - fy, gz = 1.f - fz;
  const float w000 = gx * gy * gz, w100 = fx * gy * gz, w010 = gx * fy * gz, w110 = fx * fy * gz;
  const float w001 = gx * gy * fz, w101 = fx * gy * fz, w011 = gx * fy * fz, w111 = fx * fy * fz;
  ux += w000 * c000.x + w100 * c100.x + w010 * c010.x + w110 * c110.x + w001 * c001.x + w101 * c101.x +
        w011 * c011.x + w111 * c111.x;
  uy += w000 * c000.y + w100 * c100.y + w010 * c010.y + w110 * c110.y + w001 * c001.y + w101 * c101.y +
        w011 * c011.y + w111 * c111.y;
  uz += w000 * c000.z + w100 * c100.z + w010 * c010.z + w110 * c110.z + w001 * c001.z + w101 * c101.z +
        w011 * c011.z + w111 * c111.z;
}

// The payload averaged over the levels at p (Eq. 1): a = the displacement (or z of the
// Cayley payload), t = the Cayley translation (zero for the displacement payload)
__device__ void eval_payload(const Job& J, float px, float py, float pz, float3& a, float3& t) {
  float ax = 0.f, ay = 0.f, az = 0.f, tx = 0.f, ty = 0.f, tz = 0.f;
  for (int l = 0; l < J.L; ++l) {
    const Level& lv = J.lev[l];
    const LevelCoord c = level_coord(J, lv, px, py, pz);
    level_add(c, lv.theta, ax, ay, az);
    if (J.C == 6) level_add(c, lv.theta_t, tx, ty, tz);
  }
  const float invL = 1.f / (float)J.L;
  a = make_float3(ax * invL, ay * invL, az * invL);
  t = make_float3(tx * invL, ty * invL, tz * invL);
}

// the deformed position of x (Sec. 3.3): x + u(x), or R(z(x)) x + t(x) with the Cayley
// payload (then also z and u = (I - Z)^{-1} x for the backward)
__device__ __forceinline__ float3 deform_point(const Job& J, float3 x, float3& z, float3& u) {
  float3 a, t;
  eval_payload(J, x.x, x.y, x.z, a, t);
  if (J.C != 6) return make_float3(x.x + a.x, x.y + a.y, x.z + a.z);
  z = a;
  u = cayley_u(z, x);
  return make_float3(2.f * u.x - x.x + t.x, 2.f * u.y - x.y + t.y, 2.f * u.z - x.z + t.z);
}

// y = x + u(x) on Q, in the slot order of the moving tree: a block takes one node, so the lanes of
// a warp interpolate between the same or neighbouring grid vertices, and stores the node's points
// and boxes on the way; clears the point's fixed-point reverse-Chamfer accumulator.  The thread of
// a job's first slot also starts the job's step (job_bump; bump 0: none).
__global__ void __launch_bounds__(NODE) k_interp(const Plan* __restrict__ P, int bump) {
  const int nj = P->n_jobs;
  const int total = P->pre[ST_NODE][nj];
  for (int it = blockIdx.x; it < total; it += gridDim.x) {
    const int j = find_job(P->pre[ST_NODE], nj, it);
    const Job& J = *P->jobs[j];
    const int nd = it - P->pre[ST_NODE][j];
    const int slot = nd * NODE + threadIdx.x;
    if (bump && slot == 0) job_bump(J, bump);
    const float4 x = __ldg(J.xs + slot);
    const int p = __float_as_int(x.w);
    float3 yy = make_float3(0.f, 0.f, 0.f);
    if (p >= 0) {
      float3 z, u;
      yy = deform_point(J, make_float3(x.x, x.y, x.z), z, u);
      J.y[p] = make_float4(yy.x, yy.y, yy.z, 0.f);
      if (J.C == 6) {
        J.zq[p] = make_float4(z.x, z.y, z.z, 0.f);
        J.uq[p] = make_float4(u.x, u.y, u.z, 0.f);
      }
      J.acc[3 * p + 0] = 0;
      J.acc[3 * p + 1] = 0;
      J.acc[3 * p + 2] = 0;
    }
    store_node(J.mov, nd, yy.x, yy.y, yy.z, p >= 0);
  }
}

// boxes of 32 nodes [node0 + 32 s, node0 + nodes) of a set, by one warp
__device__ __forceinline__ void super_box(const Tree& T, const SetRange& r, int s) {
  const int lane = threadIdx.x & 31;
  const float inf = __int_as_float(0x7f800000);
  const int nd = 32 * s + lane;
  float4 a = make_float4(inf, inf, inf, -inf), c = make_float4(-inf, -inf, 0.f, 0.f);
  if (nd < r.nodes) {
    a = T.nbox[2 * (r.node0 + nd)];
    c = T.nbox[2 * (r.node0 + nd) + 1];
  }
  float b[6] = {a.x, a.y, a.z, a.w, c.x, c.y};
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float v = __shfl_xor_sync(0xffffffffu, b[k], o);
      b[k] = k < 3 ? fminf(b[k], v) : fmaxf(b[k], v);
    }
  if (lane == 0) {
    T.sbox[2 * (r.super0 + s)] = make_float4(b[0], b[1], b[2], b[3]);
    T.sbox[2 * (r.super0 + s) + 1] = make_float4(b[4], b[5], 0.f, 0.f);
  }
}

// super-node boxes of the moving trees, a warp each
__global__ void __launch_bounds__(64) k_boxes(const Plan* __restrict__ P) {
  const int nj = P->n_jobs;
  const int total = P->pre[ST_SUPER][nj];
  for (int it = blockIdx.x * 2 + (threadIdx.x >> 5); it < total; it += gridDim.x * 2) {
    const int j = find_job(P->pre[ST_SUPER], nj, it);
    const Job& J = *P->jobs[j];
    const int s = it - P->pre[ST_SUPER][j];
    const SetRange r0 = mov_set(J, 0);
    if (s < r0.supers) super_box(J.mov, r0, s);
    else super_box(J.mov, mov_set(J, 1), s - r0.supers);
  }
}

// ------------------------------------------------------------------------------ (c) isometry

// |a - b| with explicit rounding so every kernel computes it bit-identically
__device__ __forceinline__ float edge_len(float4 a, float4 b) {
  return __fsqrt_rn(sqdist(a.x, a.y, a.z, b.x, b.y, b.z));
}

// per edge: |r| with r = |y_i - y_j| - e_prev, and sgn(r)(y_i - y_j)/(|y_i - y_j| |E|)
// (Sec. 3.4; sgn(0) = 0, zero-length edges contribute no gradient)
__global__ void k_iso_edges(const Plan* __restrict__ P) {
  const int nj = P->n_jobs;
  const int total = P->pre[ST_E][nj];
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < total; it += gridDim.x * blockDim.x) {
    const int j = find_job(P->pre[ST_E], nj, it);
    const Job& J = *P->jobs[j];
    const int e = it - P->pre[ST_E][j];
    const int2 ij = J.edges[e];
    const float4 a = J.y[ij.x], b = J.y[ij.y];
    const float len = edge_len(a, b);
    const float r = len - J.e_prev[e];
    J.loss_iso[e] = fabsf(r);
    float c = 0.f;
    if (len > 0.f && r != 0.f) c = copysignf(1.f, r) / (len * (float)J.E);
    J.edge_d[e] = make_float4(c * (a.x - b.x), c * (a.y - b.y), c * (a.z - b.z), 0.f);
  }
}

// dLoss/dy = forward Chamfer term + (w/M) * reverse Chamfer sums + w_iso * isometry
// gradient gathered over the vertex's edges in a fixed order.
__global__ void k_assemble(const Plan* __restrict__ P) {
  const int nj = P->n_jobs;
  const int total = P->pre[ST_Q][nj];
  for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < total; it += gridDim.x * blockDim.x) {
    const int j = find_job(P->pre[ST_Q], nj, it);
    const Job& J = *P->jobs[j];
    const int p = it - P->pre[ST_Q][j];
    float4 g = J.gfwd[p];
    const float wr = (p < J.V ? J.w_mesh : J.w_pts) / (float)J.M;
    g.x += wr * from_fx(J.acc[3 * p + 0]);
    g.y += wr * from_fx(J.acc[3 * p + 1]);
    g.z += wr * from_fx(J.acc[3 * p + 2]);
    if (p < J.V && J.w_iso != 0.f) {
      float ix = 0.f, iy = 0.f, iz = 0.f;
      const int k1 = J.v2e_ptr[p + 1];
      for (int k = J.v2e_ptr[p]; k < k1; k += 8) {  // 8 edges at a time, loads before sums
        int ent[8];
        float4 d[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) ent[u] = k + u < k1 ? __ldg(J.v2e + k + u) : -1;
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (ent[u] >= 0) d[u] = __ldg(J.edge_d + (ent[u] >> 1));
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (ent[u] < 0) break;
          if (ent[u] & 1) { ix -= d[u].x; iy -= d[u].y; iz -= d[u].z; }
          else { ix += d[u].x; iy += d[u].y; iz += d[u].z; }
        }
      }
      g.x += J.w_iso * ix;
      g.y += J.w_iso * iy;
      g.z += J.w_iso * iz;
    }
    J.gy[p] = g;
    const int slot = J.slot_of[p];
    J.gys[slot] = g;
    float gm = fmaxf(fabsf(g.x), fmaxf(fabsf(g.y), fabsf(g.z)));
    if (J.C == 6) {  // the point's gradient with respect to its averaged Cayley z
      const float4 z4 = J.zq[p], u4 = J.uq[p];
      const float3 gzv = cayley_grad_z(make_float3(z4.x, z4.y, z4.z), make_float3(u4.x, u4.y, u4.z),
                                       make_float3(g.x, g.y, g.z));
      J.gz[slot] = make_float4(gzv.x, gzv.y, gzv.z, 0.f);
      gm = fmaxf(gm, fmaxf(fabsf(gzv.x), fmaxf(fabsf(gzv.y), fabsf(gzv.z))));
    }
    // running bound on the point gradients of the job (order-independent max, one atomic per
    // job per warp); it sets the adjoint's fixed-point scale
    unsigned bits = __float_as_uint(gm);
    if (!(gm <= 3.0e38f)) bits = 0x7f800000u;
    const unsigned act = __activemask();
    const unsigned same = __match_any_sync(act, j);
    const unsigned m = __reduce_max_sync(same, bits);
    if ((threadIdx.x & 31) == __ffs(same) - 1) atomicMax(J.gmax, m);
  }
}

// ------------------------------------------------------------------------------ loss

// Loss record.  The per-query and per-edge terms of a job form one virtual array
// [phi fwd (Q) | phi rev set 0 (M) | phi rev set 1 (M, if N > 0) | |r| (E)], cut into fixed chunks of
// LOSS_CHUNK; each chunk is summed by one block in a fixed fp32 tree per term, and a second
// kernel adds a job's chunk partials in order in FP64.  The partition depends only on the
// job, so a job's loss is bitwise the same alone or in a batch.
__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  float t = 0.f;
  if (w == 0) {
    t = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;  // valid in thread 0
}

__global__ void __launch_bounds__(256) k_loss_chunks(const Plan* __restrict__ P) {
  __shared__ float red[32];
  const int nj = P->n_jobs;
  const int total = P->pre[ST_LOSSCH][nj];
  for (int it = blockIdx.x; it < total; it += gridDim.x) {
    const int j = find_job(P->pre[ST_LOSSCH], nj, it);
    const Job& J = *P->jobs[j];
    const int c = it - P->pre[ST_LOSSCH][j];
    const int b0 = c * LOSS_CHUNK;
    const int Q = J.Q, V = J.V, M = J.M;
    const int rev_end = Q + (J.N > 0 ? 2 : 1) * M;
    const int n_all = rev_end + J.E;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f, s4 = 0.f;
    for (int i = b0 + threadIdx.x; i < min(b0 + LOSS_CHUNK, n_all); i += blockDim.x) {
      if (i < V) s0 += J.loss_fwd[i];
      else if (i < Q) s1 += J.loss_fwd[i];
      else if (i < Q + M) s2 += J.loss_rev[i - Q];
      else if (i < rev_end) s3 += J.loss_rev[i - Q];
      else s4 += J.loss_iso[i - rev_end];
    }
    const float t0 = block_sum(s0, red), t1 = block_sum(s1, red), t2 = block_sum(s2, red);
    const float t3 = block_sum(s3, red), t4 = block_sum(s4, red);
    if (threadIdx.x == 0) {
      float* o = J.loss_part + 5 * c;
      o[0] = t0; o[1] = t1; o[2] = t2; o[3] = t3; o[4] = t4;
    }
  }
}

__global__ void __launch_bounds__(256) k_loss_final(const Plan* __restrict__ P) {
  __shared__ float red[32];
  const int nj = P->n_jobs;
  for (int j = blockIdx.x; j < nj; j += gridDim.x) {
    const Job& J = *P->jobs[j];
    const int nch = (J.Q + (J.N > 0 ? 2 : 1) * J.M + J.E + LOSS_CHUNK - 1) / LOSS_CHUNK;
    float s[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
    for (int c = threadIdx.x; c < nch; c += blockDim.x) {
#pragma unroll
      for (int k = 0; k < 5; ++k) s[k] += J.loss_part[5 * c + k];
    }
    double t[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) t[k] = (double)block_sum(s[k], red);  // all terms are >= 0
    if (threadIdx.x == 0) {
      const double cdm = t[0] / J.V + t[2] / J.M;
      const double cdp = J.N > 0 ? t[1] / (J.Q - J.V) + t[3] / J.M : 0.0;
      const double iso = J.E > 0 ? t[4] / J.E : 0.0;
      const double tot = (double)J.w_mesh * cdm + (double)J.w_pts * cdp + (double)J.w_iso * iso;
      J.loss[0] = tot;
      J.loss[1] = cdm;
      J.loss[2] = cdp;
      J.loss[3] = iso;
      if (!isfinite(tot)) *J.status |= 1;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------ per frame

__global__ void k_pack4(const float* __restrict__ in, float4* __restrict__ out, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = make_float4(in[3 * i], in[3 * i + 1], in[3 * i + 2], 0.f);
}

__global__ void k_unpack4(const float4* __restrict__ in, float* __restrict__ out, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float4 v = in[i];
    out[3 * i] = v.x;
    out[3 * i + 1] = v.y;
    out[3 * i + 2] = v.z;
  }
}

__global__ void k_check_finite(const float* __restrict__ in, int n, int* flag) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    if (!isfinite(in[i])) atomicOr(flag, 1);
}

// Q = X_{t-1} u P_{t-1}; rest lengths e_prev from X_{t-1} (same expression as k_iso_edges
// so that zero grids give r == 0 exactly).
__global__ void k_frame_points(Job* J) {
  const int Q = J->Q, V = J->V;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < Q; p += gridDim.x * blockDim.x)
    J->x[p] = p < V ? J->verts4[p] : J->src4[p - V];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < J->E; e += gridDim.x * blockDim.x) {
    const int2 ij = J->edges[e];
    J->e_prev[e] = edge_len(J->verts4[ij.x], J->verts4[ij.y]);
  }
}

// Tree builds (per frame), both trees in each launch: cell keys and counts, scatter of the indices into
// slot order.  i < M: target i; else moving point i - M.
__global__ void k_tree_keys(Job* J) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < J->M + J->Q; i += gridDim.x * blockDim.x) {
    const bool t = i < J->M;
    const int p = t ? i : i - J->M;
    const float4 x = t ? J->tgt4[p] : J->x[p];
    const Tree& T = t ? J->tgt : J->mov;
    const int key = cell_key(T, x.x, x.y, x.z, t || p < J->V ? 0 : 1);
    T.keys[p] = key;
    atomicAdd(&T.hist[key], 1);
  }
}

__global__ void k_tree_scatter(Job* J) {
  const SetRange r0 = mov_set(*J, 0), r1 = mov_set(*J, 1);
  const int pad0 = r0.nodes * NODE - r0.n, pad1 = r1.nodes * NODE - r1.n;
  const int M = J->M, Q = J->Q;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M + Q + pad0 + pad1; i += gridDim.x * blockDim.x) {
    if (i < M + Q) {
      const bool t = i < M;
      const int p = t ? i : i - M;
      const Tree& T = t ? J->tgt : J->mov;
      const int key = T.keys[p];
      const int pos = T.off[key] + atomicSub(&T.hist[key], 1) - 1;
      const int slot = t || p < J->V ? pos : r1.slot0 + pos - J->V;
      T.perm[slot] = p;
      if (!t) {
        const float4 x = J->x[p];
        J->xs[slot] = make_float4(x.x, x.y, x.z, __int_as_float(p));
        J->slot_of[p] = slot;
      }
    } else {  // padding of the moving sets' last nodes
      const int k = i - M - Q;
      const int slot = k < pad0 ? r0.n + k : r1.slot0 + r1.n + k - pad0;
      J->xs[slot] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
      J->mov.perm[slot] = -1;
    }
  }
}

// target points and boxes, a block per node
__global__ void __launch_bounds__(NODE) k_tgt_nodes(Job* J) {
  const int nodes = (J->M + NODE - 1) / NODE;
  for (int nd = blockIdx.x; nd < nodes; nd += gridDim.x) {
    const int slot = nd * NODE + threadIdx.x;
    const bool in = slot < J->M;
    if (!in) J->tgt.perm[slot] = -1;
    const float4 t = in ? J->tgt4[J->tgt.perm[slot]] : make_float4(0.f, 0.f, 0.f, 0.f);
    store_node(J->tgt, nd, t.x, t.y, t.z, in);
  }
}

__global__ void __launch_bounds__(32) k_tgt_boxes(Job* J) {
  const SetRange r = set_range(0, 0, J->M);
  for (int s = blockIdx.x; s < r.supers; s += gridDim.x) super_box(J->tgt, r, s);
}

// frame end: X_t = M(T_t(X_{t-1})) X_{t-1} with the final grids (Sec. 3.3)
__global__ void k_end_frame(Job* J) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < J->V; p += gridDim.x * blockDim.x) {
    const float4 x = J->x[p];
    float3 z, u;
    const float3 y = deform_point(*J, make_float3(x.x, x.y, x.z), z, u);
    J->verts4[p] = make_float4(y.x, y.y, y.z, 0.f);
  }
}

// the frame's deformation applied to arbitrary points ([n][3] float in/out, device)
__global__ void k_deform(const Job* __restrict__ J, const float* __restrict__ in, float* __restrict__ out, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    float3 z, u;
    const float3 y = deform_point(*J, make_float3(in[3 * i], in[3 * i + 1], in[3 * i + 2]), z, u);
    out[3 * i] = y.x;
    out[3 * i + 1] = y.y;
    out[3 * i + 2] = y.z;
  }
}

// ------------------------------------------------------------------------------ launchers

static inline int blocks_for(int n, int threads) { return max(1, min((n + threads - 1) / threads, 4096)); }

void launch_plan(Plan* P, cudaStream_t s) { k_plan<<<1, 256, 0, s>>>(P); }
void launch_job(const Job& job, Job* dJ, cudaStream_t s) {
  static_assert(sizeof(Job) % 4 == 0, "copied word by word");
  k_op_job<<<1, 256, 0, s>>>(job, dJ, nullptr);
}
void launch_op_plan(const Job& job, Job* dJ, Plan* dP, cudaStream_t s) {
  k_op_job<<<1, 256, 0, s>>>(job, dJ, dP);
  launch_plan(dP, s);
}
void launch_interp(const Plan* P, int grid, cudaStream_t s, int bump) { k_interp<<<grid, 256, 0, s>>>(P, bump); }
void launch_boxes(const Plan* P, int grid, cudaStream_t s) { k_boxes<<<grid, 64, 0, s>>>(P); }
void launch_iso_edges(const Plan* P, int grid, cudaStream_t s) { k_iso_edges<<<grid, 256, 0, s>>>(P); }
void launch_assemble(const Plan* P, int grid, cudaStream_t s) { k_assemble<<<grid, 256, 0, s>>>(P); }
void launch_loss(const Plan* P, int chunks, int jobs, cudaStream_t s) {
  k_loss_chunks<<<chunks, 256, 0, s>>>(P);
  k_loss_final<<<jobs, 256, 0, s>>>(P);
}

void launch_pack4(const float* in, float4* out, int n, cudaStream_t s) {
  k_pack4<<<blocks_for(n, 256), 256, 0, s>>>(in, out, n);
}
void launch_unpack4(const float4* in, float* out, int n, cudaStream_t s) {
  k_unpack4<<<blocks_for(n, 256), 256, 0, s>>>(in, out, n);
}
void launch_check_finite(const float* in, int n, int* flag, cudaStream_t s) {
  k_check_finite<<<blocks_for(n, 256), 256, 0, s>>>(in, n, flag);
}
void launch_frame_points(Job* J, int Q, int E, cudaStream_t s) {
  k_frame_points<<<blocks_for(max(Q, E), 256), 256, 0, s>>>(J);
}
void launch_end_frame(Job* J, int V, cudaStream_t s) { k_end_frame<<<blocks_for(V, 256), 256, 0, s>>>(J); }
void launch_deform(const Job* J, const float* in, float* out, int n, cudaStream_t s) {
  k_deform<<<blocks_for(n, 256), 256, 0, s>>>(J, in, out, n);
}

// channel-planar [C][n3] -> interleaved [n3][C]
__global__ void k_soa_to_aos(const float* __restrict__ in, float* __restrict__ out, int n3, int C) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += gridDim.x * blockDim.x)
    for (int c = 0; c < C; ++c) out[(size_t)C * i + c] = in[(size_t)c * n3 + i];
}
void launch_soa_to_aos(const float* in, float* out, int n3, cudaStream_t s, int C) {
  k_soa_to_aos<<<blocks_for(n3, 256), 256, 0, s>>>(in, out, n3, C);
}

// level values [n3][C] <-> the float4 arrays of a level (theta; theta_t holds channels 3..5); packing
// also clears the level's Adam moments
__global__ void k_pack_theta(const float* __restrict__ in, float4* __restrict__ th, float4* __restrict__ tht,
                             float* __restrict__ m, float* __restrict__ v, int n3, int C) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += gridDim.x * blockDim.x) {
    const float* r = in + (size_t)C * i;
    th[i] = make_float4(r[0], r[1], r[2], 0.f);
    if (C == 6) tht[i] = make_float4(r[3], r[4], r[5], 0.f);
    for (int c = 0; c < C; ++c) m[(size_t)c * n3 + i] = v[(size_t)c * n3 + i] = 0.f;
  }
}
__global__ void k_unpack_theta(const float4* __restrict__ th, const float4* __restrict__ tht, float* __restrict__ out,
                               int n3, int C) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += gridDim.x * blockDim.x) {
    float* r = out + (size_t)C * i;
    const float4 a = th[i];
    r[0] = a.x; r[1] = a.y; r[2] = a.z;
    if (C == 6) {
      const float4 b = tht[i];
      r[3] = b.x; r[4] = b.y; r[5] = b.z;
    }
  }
}
void launch_pack_theta(const float* in, float4* th, float4* tht, float* m, float* v, int n3, int C, cudaStream_t s) {
  k_pack_theta<<<blocks_for(n3, 256), 256, 0, s>>>(in, th, tht, m, v, n3, C);
}
void launch_unpack_theta(const float4* th, const float4* tht, float* out, int n3, int C, cudaStream_t s) {
  k_unpack_theta<<<blocks_for(n3, 256), 256, 0, s>>>(th, tht, out, n3, C);
}

// both trees of the frame: keys + counts, exclusive scans, scatter; the targets' points and boxes (the
// moving points' come with the interpolation)
void launch_tree_build(Job* J, const Job& hJ, cudaStream_t s) {
  const int n = hJ.M + hJ.Q;
  k_tree_keys<<<blocks_for(n, 256), 256, 0, s>>>(J);
  launch_scan(ScanSeg{hJ.tgt.hist, hJ.tgt.off, 1 << (3 * hJ.tgt.bits), hJ.tgt.csum},
              ScanSeg{hJ.mov.hist, hJ.mov.off, 2 << (3 * hJ.mov.bits), hJ.mov.csum}, s);
  k_tree_scatter<<<blocks_for(n + 2 * NODE, 256), 256, 0, s>>>(J);
  const SetRange r = set_range(0, 0, hJ.M);
  k_tgt_nodes<<<min(r.nodes, 4096), NODE, 0, s>>>(J);
  k_tgt_boxes<<<min(r.supers, 4096), 32, 0, s>>>(J);
}

}  // namespace pdg
