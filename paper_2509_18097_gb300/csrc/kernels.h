// Host-side launchers of the libpdg kernels (each defined next to its kernels).
#pragma once
#include <algorithm>
#include <vector>

#include "pdg_internal.cuh"

namespace pdg {

// per step (plan-driven; `grid` = blocks of the persistent launch)
void launch_plan(Plan* P, cudaStream_t s);
// a job's record, and with it a plan for it alone, from the launch's arguments (nothing is copied from
// host memory)
void launch_job(const Job& job, Job* dJ, cudaStream_t s);
void launch_op_plan(const Job& job, Job* dJ, Plan* dP, cudaStream_t s);
void launch_interp(const Plan* P, int grid, cudaStream_t s, int bump);
void launch_boxes(const Plan* P, int grid, cudaStream_t s);
// set < 0: the moving points' searches in the target tree, else the targets' in the tree of a moving
// set; sub: lanes per query (2 or 8); count: the instance that counts candidates and exact ties
void launch_nn(const Plan* P, int grid, cudaStream_t s, int set, int sub, bool count);
void launch_iso_edges(const Plan* P, int grid, cudaStream_t s);
void launch_assemble(const Plan* P, int grid, cudaStream_t s);
void launch_adjoint_rows(const Plan* P, int grid, cudaStream_t s);
void launch_adjoint(const Plan* P, int grid, cudaStream_t s);
// line path (256 and sizes with a factor 3); nmax: the largest level it takes in the plan
enum YzPass { YZ_FWD = 0, YZ_Z, YZ_INV };
void launch_sobolev_x(const Plan* P, int grid, int nmax, bool fwd, cudaStream_t s);
void launch_sobolev_yz(const Plan* P, int grid, int nmax, int pass, cudaStream_t s);
void launch_sobolev_plane(const Plan* P, int grid, int nmax, cudaStream_t s, int part, bool ext);
void launch_loss(const Plan* P, int chunks, int jobs, cudaStream_t s);

// per frame / per call (one job)
void launch_pack4(const float* in, float4* out, int n, cudaStream_t s);
void launch_unpack4(const float4* in, float* out, int n, cudaStream_t s);
void launch_check_finite(const float* in, int n, int* flag, cudaStream_t s);
void launch_frame_points(Job* J, int Q, int E, cudaStream_t s);
void launch_tree_build(Job* J, const Job& hJ, cudaStream_t s);
void launch_nn_seed(Job* J, const Job& hJ, cudaStream_t s);
void launch_csr_build(Job* J, const Job& hJ, cudaStream_t s);
void launch_end_frame(Job* J, int V, cudaStream_t s);
void launch_deform(const Job* J, const float* in, float* out, int n, cudaStream_t s);

// exclusive scans of two arrays
struct ScanSeg {
  const int* in;
  int* out;   // [len + 1]
  int len;
  int* csum;  // [ceil(len / SCAN_CHUNK)]
};
void launch_scan(const ScanSeg& a, const ScanSeg& b, cudaStream_t s);
void launch_csr_scan(const Job* J, const Job& hJ, cudaStream_t s);

void sobolev_x_configure();
void sobolev_yz_configure();
void sobolev_plane_configure();
int plane_smem_bytes(int n);
int plane_smem_max(int nmax);
void launch_sobz_pivots(float* piv, int* slow, const float* mu, int n, float lam, cudaStream_t s);

// template-mesh fit (k_mesh.cu)
constexpr int MESH_WAIT = 1 << 20;  // looks at a grid barrier: about half a second
void launch_mesh_points(Job* J, int V, cudaStream_t s);
// (I + lambda L)^{-2} b by two Chebyshev solves, then Adam on x
struct MeshSolve {
  const int *ptr, *nbr;  // neighbour lists of the vertices
  const float4* b;       // right-hand side
  float4 *h, *r, *d0, *d1;
  float4 *pg;            // the result
  float4 *x, *m, *v;
  float2* coef;          // [iters] constants of the recurrence (mesh_coef)
  unsigned* bar;         // grid barrier
  int wait;              // looks at the barrier before a block gives up
  int* err;              // set when the barrier's wait ran out
  int V, iters;
  int degree;            // largest of a vertex
  float lam, inv_theta, lr, b1, b2, eps, bias1, ibias2;
};
void launch_mesh_commit(const MeshSolve& a, float4* verts, cudaStream_t s);
void mesh_coef(std::vector<float2>& coef, int iters, float emax);
// refuse: cooperative launches still to be taken as refused (test hook)
cudaError_t launch_mesh_solve(MeshSolve a, float emax, int sms, int& refuse, cudaStream_t s);

// misc conversions
void launch_soa_to_aos(const float* in, float* out, int n3, cudaStream_t s, int C = 3);
void launch_pack_theta(const float* in, float4* th, float4* tht, float* m, float* v, int n3, int C, cudaStream_t s);
void launch_unpack_theta(const float4* th, const float4* tht, float* out, int n3, int C, cudaStream_t s);

}  // namespace pdg
