// Template-mesh fit (Sec. 3.4, surface initialisation loss L_mesh = CD_R(X_0, P_0); Sec. 3.6,
// lambda = 16, lr = 1e-4): the kernels of one iteration that the frame step does not have.
// The robust Chamfer search and gradient are the step's own kernels, run on a job record
// whose query points are the mesh vertices alone (no source set, no isometry term).  The
// vertex gradient is then preconditioned by (I + lambda L)^{-2}, L the combinatorial graph
// Laplacian of the mesh edges, by two Chebyshev solves (no inner products), and Adam moves the
// vertices: both in one cooperative launch (k_mesh_solve), or with a launch per Chebyshev iteration
// where that does not fit.
#include "kernels.h"

namespace pdg {

// y = x for the mesh vertices (the query points of the fit), their tree nodes (a block each, in
// the slot order of the fit's start), cleared reverse-Chamfer accumulators; the first thread
// clears the step's counters.
__global__ void __launch_bounds__(NODE) k_mesh_points(Job* __restrict__ Jp) {
  const Job& J = *Jp;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *J.gmax = 0u;
    J.counters[CNT_NN_CANDIDATES] = 0ull;
    J.counters[CNT_NN_TIES] = 0ull;
  }
  const int nodes = (J.V + NODE - 1) / NODE;
  for (int nd = blockIdx.x; nd < nodes; nd += gridDim.x) {
    const int p = J.mov.perm[nd * NODE + threadIdx.x];
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p >= 0) {
      x = J.x[p];
      J.y[p] = make_float4(x.x, x.y, x.z, 0.f);
      J.acc[3 * p + 0] = 0;
      J.acc[3 * p + 1] = 0;
      J.acc[3 * p + 2] = 0;
    }
    store_node(J.mov, nd, x.x, x.y, x.z, p >= 0);
  }
}

// Chebyshev iteration for A h = b, A = I + lambda L (symmetric, eigenvalues in [1, emax]),
// as the three-term recurrence: h_{k+1} = h_k + d_k, r_{k+1} = r_k - A d_k,
// d_{k+1} = c1 d_k + c2 r_{k+1}, started from h_0 = 0, r_0 = b, d_0 = b / theta.
// Set-up of the recurrence.
__global__ void k_cheb_init(const float4* __restrict__ b, float4* __restrict__ h, float4* __restrict__ r,
                            float4* __restrict__ d, int V, float inv_theta) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < V; i += gridDim.x * blockDim.x) {
    const float4 v = b[i];
    h[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    r[i] = make_float4(v.x, v.y, v.z, 0.f);
    d[i] = make_float4(v.x * inv_theta, v.y * inv_theta, v.z * inv_theta, 0.f);
  }
}

// One iteration: (A d)_i = d_i + lambda sum_{j ~ i} (d_i - d_j) over the vertex's edges (the
// neighbour lists of the context); d is read from
// `din` (complete from the previous launch) and the next d written to `dout`.
__global__ void k_cheb_iter(const int* __restrict__ ptr, const int* __restrict__ nbr, const float4* __restrict__ din, float4* __restrict__ dout, float4* __restrict__ h,
                            float4* __restrict__ r, int V, float lam, float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < V; i += gridDim.x * blockDim.x) {
    const float4 di = din[i];
    float lx = 0.f, ly = 0.f, lz = 0.f;
    for (int k = __ldg(ptr + i); k < __ldg(ptr + i + 1); ++k) {
      const float4 dj = din[__ldg(nbr + k)];
      lx += di.x - dj.x;
      ly += di.y - dj.y;
      lz += di.z - dj.z;
    }
    const float ax = di.x + lam * lx, ay = di.y + lam * ly, az = di.z + lam * lz;
    float4 hi = h[i], ri = r[i];
    hi.x += di.x; hi.y += di.y; hi.z += di.z;
    ri.x -= ax; ri.y -= ay; ri.z -= az;
    h[i] = hi;
    r[i] = ri;
    dout[i] = make_float4(c1 * di.x + c2 * ri.x, c1 * di.y + c2 * ri.y, c1 * di.z + c2 * ri.z, 0.f);
  }
}

// Adam (PyTorch semantics) on the mesh vertices with the preconditioned gradient g;
// bias1 = 1 / (1 - beta1^k), ibias2 = 1 / sqrt(1 - beta2^k)
__device__ __forceinline__ void adam_vertex(float4* x, float4 gi, float4* m, float4* v, int i, float lr, float b1,
                                            float b2, float eps, float bias1, float ibias2) {
  float4 mi = m[i], vi = v[i], xi = x[i];
  const float gg[3] = {gi.x, gi.y, gi.z};
  float* mm = &mi.x;
  float* vv = &vi.x;
  float* xx = &xi.x;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    mm[c] = b1 * mm[c] + (1.f - b1) * gg[c];
    vv[c] = b2 * vv[c] + (1.f - b2) * gg[c] * gg[c];
    xx[c] -= lr * bias1 * mm[c] / (sqrtf(vv[c]) * ibias2 + eps);
  }
  m[i] = mi;
  v[i] = vi;
  x[i] = xi;
}

__global__ void k_mesh_adam(float4* __restrict__ x, const float4* __restrict__ g, float4* __restrict__ m,
                            float4* __restrict__ v, int V, float lr, float b1, float b2, float eps, float bias1,
                            float ibias2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < V; i += gridDim.x * blockDim.x)
    adam_vertex(x, g[i], m, v, i, lr, b1, b2, eps, bias1, ibias2);
}

// ------------------------------------------------------------------------------ in one launch

// Both solves and Adam in one cooperative launch.  A thread keeps its K vertices' h, r and d in
// registers for all iterations; only d crosses threads, through two buffers in L2 and a barrier of
// the grid's blocks (at most one per SM) after each write; a vertex's neighbours are loaded together.
// What bounds it: the latency of the barrier and of one gather from L2, 1.9 us an iteration on 50 412
// vertices (a launch per iteration: 6.5 us, 270 of them).  Neighbours loaded one after another: 2.65
// us; 1024 threads a block (half the blocks, 64 registers): 3.4 us; 384 threads: the same.  A vertex of
// 518 edges on 50 400 vertices: 40 us an iteration (its later neighbours one after another: 82; a launch
// per iteration: 96).
constexpr int MS_THREADS = 512;

// All blocks of the grid (co-resident: cooperative launch).  False after `limit` looks at the count
// (MESH_WAIT: about half a second): the kernel then gives up and the caller reports it.
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned target, int limit, int* err) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    unsigned seen = 0;
    int looks = 0;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
    } while (seen < target && ++looks < limit);
    ok = seen >= target;
    if (!ok) atomicExch(err, 1);
  }
  __syncthreads();
  return ok;
}

template <int K>
__global__ void __launch_bounds__(MS_THREADS) k_mesh_solve(const MeshSolve a) {
  constexpr int NB = K <= 2 ? 8 : 4;  // as many as leave no register spilled
  const int V = a.V, base = blockIdx.x * (MS_THREADS * K) + threadIdx.x;
  float h[K][3], r[K][3], d[K][3];
  int p0[K], p1[K];
  int nb[K][NB];  // a vertex's first neighbours
  unsigned phase = 0;
  float4* din = a.d0;
  float4* dout = a.d1;
  // some block gave up: leave the vertices as they are (the whole block decides alike)
  if (__syncthreads_or(*reinterpret_cast<volatile int*>(a.err))) return;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = base + k * MS_THREADS;
    p0[k] = i < V ? __ldg(a.ptr + i) : 0;
    p1[k] = i < V ? __ldg(a.ptr + i + 1) : 0;
#pragma unroll
    for (int e = 0; e < NB; ++e) nb[k][e] = p0[k] + e < p1[k] ? __ldg(a.nbr + p0[k] + e) : -1;
    const float4 g = i < V ? a.b[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    h[k][0] = g.x;
    h[k][1] = g.y;
    h[k][2] = g.z;
  }
  for (int solve = 0; solve < 2; ++solve) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int i = base + k * MS_THREADS;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        r[k][c] = h[k][c];
        h[k][c] = 0.f;
        d[k][c] = r[k][c] * a.inv_theta;
      }
      if (i < V) din[i] = make_float4(d[k][0], d[k][1], d[k][2], 0.f);
    }
    if (!grid_barrier(a.bar, ++phase * gridDim.x, a.wait, a.err)) return;
    for (int it = 0; it < a.iters; ++it) {
      const float2 co = __ldg(a.coef + it);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int i = base + k * MS_THREADS;
        float l[3] = {0.f, 0.f, 0.f};
        float4 dj[NB];  // all in flight together
#pragma unroll
        for (int e = 0; e < NB; ++e)
          if (nb[k][e] >= 0) dj[e] = __ldcg(din + nb[k][e]);
#pragma unroll
        for (int e = 0; e < NB; ++e)
          if (nb[k][e] >= 0) {
            l[0] += d[k][0] - dj[e].x;
            l[1] += d[k][1] - dj[e].y;
            l[2] += d[k][2] - dj[e].z;
          }
#pragma unroll 1
        for (int e0 = p0[k] + NB; e0 < p1[k]; e0 += NB) {  // the others, as many at a time
          int id[NB];
#pragma unroll
          for (int e = 0; e < NB; ++e) id[e] = e0 + e < p1[k] ? __ldg(a.nbr + e0 + e) : -1;
#pragma unroll
          for (int e = 0; e < NB; ++e)
            if (id[e] >= 0) dj[e] = __ldcg(din + id[e]);
#pragma unroll
          for (int e = 0; e < NB; ++e)
            if (id[e] >= 0) {
              l[0] += d[k][0] - dj[e].x;
              l[1] += d[k][1] - dj[e].y;
              l[2] += d[k][2] - dj[e].z;
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          h[k][c] += d[k][c];
          r[k][c] -= d[k][c] + a.lam * l[c];
          d[k][c] = co.x * d[k][c] + co.y * r[k][c];
        }
        if (i < V && it + 1 < a.iters) dout[i] = make_float4(d[k][0], d[k][1], d[k][2], 0.f);
      }
      float4* t = din;
      din = dout;
      dout = t;
      if (it + 1 < a.iters && !grid_barrier(a.bar, ++phase * gridDim.x, a.wait, a.err)) return;
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = base + k * MS_THREADS;
    if (i >= V) break;
    const float4 g = make_float4(h[k][0], h[k][1], h[k][2], 0.f);
    a.pg[i] = g;
    adam_vertex(a.x, g, a.m, a.v, i, a.lr, a.b1, a.b2, a.eps, a.bias1, a.ibias2);
  }
}

// The fitted vertices become the template, unless a solve gave up: blocks give up one by one, so some
// of that iteration may have moved their vertices.
__global__ void k_mesh_commit(const float4* __restrict__ x, float4* __restrict__ verts, int V, const int* __restrict__ err) {
  if (*err) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < V; i += gridDim.x * blockDim.x) verts[i] = x[i];
}

static inline int mesh_blocks(int n) { return max(1, min((n + 255) / 256, 4096)); }

void launch_mesh_points(Job* J, int V, cudaStream_t s) { k_mesh_points<<<mesh_blocks(V), NODE, 0, s>>>(J); }

void launch_mesh_commit(const MeshSolve& a, float4* verts, cudaStream_t s) {
  k_mesh_commit<<<mesh_blocks(a.V), 256, 0, s>>>(a.x, verts, a.V, a.err);
}

static void launch_cheb_solve(const MeshSolve& a, const float4* b, float4* h, double theta, double delta, cudaStream_t s) {
  const int nb = mesh_blocks(a.V);
  k_cheb_init<<<nb, 256, 0, s>>>(b, h, a.r, a.d0, a.V, a.inv_theta);
  if (delta <= 0.0) {  // lambda = 0: A = I, the set-up already holds h + d = b after one update
    k_cheb_iter<<<nb, 256, 0, s>>>(a.ptr, a.nbr, a.d0, a.d1, h, a.r, a.V, 0.f, 0.f, 0.f);
    return;
  }
  const double sigma = theta / delta;
  double rho = 1.0 / sigma;
  float4* din = a.d0;
  float4* dout = a.d1;
  for (int k = 0; k < a.iters; ++k) {
    const double rho_n = 1.0 / (2.0 * sigma - rho);
    k_cheb_iter<<<nb, 256, 0, s>>>(a.ptr, a.nbr, din, dout, h, a.r, a.V, a.lam, (float)(rho_n * rho),
                                   (float)(2.0 * rho_n / delta));
    rho = rho_n;
    std::swap(din, dout);
  }
}

// Vertices per thread of the one-launch form: the fewest that leave at most a block per SM (0: the
// mesh is too large for it, or has a vertex of so many edges that the others' wait at the barrier
// could run out while its thread walks them: 0.08 us an edge, so 4096 take 0.3 ms of about 500, where
// a launch per iteration takes 0.5).
constexpr int MS_DEGREE = 4096;
static int mesh_solve_k(int V, int degree, int sms) {
  if (degree > MS_DEGREE) return 0;
  for (int k = 1; k <= 4; k *= 2)
    if ((V + MS_THREADS * k - 1) / (MS_THREADS * k) <= sms) return k;
  return 0;
}

template <int K>
static cudaError_t launch_mesh_coop(MeshSolve a, cudaStream_t s) {
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)k_mesh_solve<K>, dim3((a.V + MS_THREADS * K - 1) / (MS_THREADS * K)),
                                     dim3(MS_THREADS), args, 0, s);
}

// the device will not hold the grid at once (fewer SMs for this context than the device has)
static bool coop_refused(cudaError_t e) {
  return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported || e == cudaErrorLaunchOutOfResources;
}

// the constants of the recurrence, c1 and c2 of each iteration (lambda = 0: A = I, one iteration)
void mesh_coef(std::vector<float2>& coef, int iters, float emax) {
  const double theta = 0.5 * (emax + 1.0), delta = 0.5 * (emax - 1.0);
  coef.assign(iters, make_float2(0.f, 0.f));
  if (delta <= 0.0) return;
  const double sigma = theta / delta;
  double rho = 1.0 / sigma;
  for (auto& c : coef) {
    const double rho_n = 1.0 / (2.0 * sigma - rho);
    c = make_float2((float)(rho_n * rho), (float)(2.0 * rho_n / delta));
    rho = rho_n;
  }
}

cudaError_t launch_mesh_solve(MeshSolve a, float emax, int sms, int& refuse, cudaStream_t s) {
  // Chebyshev constants for the interval [1, emax] (theta its centre, delta its half-width)
  const double theta = 0.5 * (emax + 1.0), delta = 0.5 * (emax - 1.0);
  a.inv_theta = (float)(1.0 / theta);
  const int k = mesh_solve_k(a.V, a.degree, sms);
  if (k > 0) {
    cudaError_t e = cudaErrorCooperativeLaunchTooLarge;
    if (refuse > 0) {
      --refuse;
    } else {
      cudaMemsetAsync(a.bar, 0, sizeof(unsigned), s);
      e = k == 1 ? launch_mesh_coop<1>(a, s) : k == 2 ? launch_mesh_coop<2>(a, s) : launch_mesh_coop<4>(a, s);
    }
    if (!coop_refused(e)) return e;
    cudaGetLastError();
  }
  launch_cheb_solve(a, a.b, a.h, theta, delta, s);
  launch_cheb_solve(a, a.h, a.pg, theta, delta, s);
  k_mesh_adam<<<mesh_blocks(a.V), 256, 0, s>>>(a.x, a.pg, a.m, a.v, a.V, a.lr, a.b1, a.b2, a.eps, a.bias1, a.ibias2);
  return cudaGetLastError();
}

}  // namespace pdg
