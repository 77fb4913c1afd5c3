// Host runtime and C ABI of libpdg: per-sequence contexts (one device arena each),
// per-frame set-up, the CUDA-graph step, batching of contexts into one graph, and
// checkpoint/resume.  See include/pdg.h for the contract of every entry point.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "kernels.h"

using namespace pdg;

namespace {

constexpr double PI = 3.14159265358979323846;

struct Arena {
  size_t off = 0;
  template <class T>
  size_t take(size_t count) {
    off = (off + 255) & ~size_t(255);
    const size_t at = off;
    off += count * sizeof(T);
    return at;
  }
};

// Cells per axis (log2) of a point tree's sort over `count` points on a surface, with about
// `per_cell` points in an occupied cell: a leaf of 8 points then spans one or two cells.
int grid_bits(long count, double per_cell = 6.0) {
  const double g = std::sqrt(std::max(count, 1L) / per_cell);
  int b = (int)std::lround(std::log2(std::max(g, 1.0)));
  return std::min(std::max(b, 2), 7);
}

// n if the line path preconditions a level of that size, else 0
int line_size(int n) { return tile_level(n) ? n : 0; }

// What the launches of a step are sized by: the largest levels, and the blocks each kernel has work
// for (at a context's capacity; for a batch the sum over its members), at most the cap beyond which
// a kernel's blocks loop over its items.  A fixed number of blocks would do, but an empty block
// still costs its launch: 4864 of them about 4 us.
struct Shape {
  int sms = 1;
  int nmax = 1;      // largest level resolution
  int nline = 0;     // largest resolution among the levels the line path preconditions (0: none)
  bool ext = false;  // the preconditioner on a caller's gradient
  enum Work {
    NODES, SUPERS,  // interpolation, upper boxes
    NNF, NNR,       // searches: warps of 32 queries, of the moving points and of the targets
    POINTS, EDGES, LOSS, JOBS,
    ROWS, ADJ,          // adjoint: blocks of long rows, blocks of warp groups
    PLANES, COLS, ADAM,  // plane path
    XT, YZ,              // line path
    N_WORK
  };
  long w[N_WORK] = {};

  // V, N points in the two moving sets, M targets, E edges
  void add_points(long V, long N, long M, long E) {
    const long vn = (V + NODE - 1) / NODE, pn = (N + NODE - 1) / NODE;
    w[NODES] += vn + pn;
    w[SUPERS] += (vn + 31) / 32 + (pn + 31) / 32;
    w[NNF] += (V + 31) / 32 + (N + 31) / 32;
    w[NNR] += (M + 31) / 32;
    w[POINTS] += V + N;
    w[EDGES] += E;
    w[LOSS] += (V + N + (N > 0 ? 2 : 1) * M + E + LOSS_CHUNK - 1) / LOSS_CHUNK;
    w[JOBS] += 1;
  }
  // a level of n vertices per axis, C channels, Q points
  void add_level(long n, long C, long Q) {
    nmax = std::max(nmax, (int)n);
    nline = std::max(nline, line_size((int)n));
    // rows (active vertices) of at most 8 Q entries: a block each from 512 entries on average, else
    // warps of up to 32 rows with at least half their lanes' entries
    const long rows = std::min(n * n * n, 8 * Q);
    w[ROWS] += std::min(rows, 8 * Q / 512 + 1);
    w[ADJ] += (8 * Q / 256 + rows / 32 + 1 + 7) / 8;
    if (line_size((int)n)) {
      w[XT] += x_tiles((int)n);
      w[YZ] += C * yz_tiles((int)n);
    } else {
      w[PLANES] += C * n;
      w[COLS] += C * ((n * n + 63) / 64);
      w[ADAM] += (n * n * n + 3) / 4;
    }
  }
  void add(const Shape& o) {  // a batch's member
    sms = o.sms;
    nmax = std::max(nmax, o.nmax);
    nline = std::max(nline, o.nline);
    for (int i = 0; i < N_WORK; ++i) w[i] += o.w[i];
  }
  // makes this cover `o` too: the larger of both in every quantity, so once covered, `o` changes nothing
  void cover(const Shape& o) {
    sms = std::max(sms, o.sms);
    nmax = std::max(nmax, o.nmax);
    nline = std::max(nline, o.nline);
    for (int i = 0; i < N_WORK; ++i) w[i] = std::max(w[i], o.w[i]);
  }
  // whether a step of this shape launches what one of `o` does.  (blocks() alone does not order shapes:
  // a small one has more lanes per query, a larger nmax a smaller cap.)
  bool same_launches(const Shape& o) const {
    bool same = sms == o.sms && nmax == o.nmax && nline == o.nline && nn_sub() == o.nn_sub() &&
                (w[PLANES] > 0) == (o.w[PLANES] > 0);
    for (int i = 0; i < N_WORK; ++i) same = same && blocks(i) == o.blocks(i);
    return same;
  }

  // Lanes per query of the searches: 8 while that leaves no more than 32 warps per SM (a warp's own
  // latency counts), else 2 (see k_nn.cu)
  int nn_sub() const { return w[NNF] + 2 * w[NNR] < 4 * sms ? 8 : 2; }
  int plane_blocks_per_sm() const { return std::max(1, std::min(8, (227 * 1024) / plane_smem_max(nmax))); }

  // blocks of a launch: what the work fills, at most the number beyond which blocks only queue
  int blocks(int i) const {
    long n = w[i], most = 8L * sms;
    switch (i) {
      case NODES: break;
      case SUPERS: n = (n + 1) / 2, most = sms; break;
      case NNF:
      case NNR: n = (n * nn_sub() + 3) / 4, most = 32L * sms; break;
      case POINTS:
      case EDGES: n = (n + 255) / 256; break;
      case LOSS: most = 2L * sms; break;
      case JOBS: most = MAXJ; break;
      case ROWS: break;
      case ADJ: most = 16L * sms; break;
      case PLANES: most = 16L * sms; break;
      case COLS: most = 32L * sms; break;
      case ADAM: n = (n + 255) / 256, most = 8L * sms * plane_blocks_per_sm(); break;
      case XT:
      case YZ: most = 256L * sms; break;
    }
    return (int)std::max(1L, std::min(n, most));
  }
};

// 1, or 2..256 with no prime factor but 2 and 3 (the line transforms are radix-2/3 FFTs)
bool valid_res(int n) {
  if (n < 1 || n > 256) return false;
  while (n % 2 == 0) n /= 2;
  while (n % 3 == 0) n /= 3;
  return n == 1;
}

// Test hook: the next `g_fail_allocs` device allocations of the library report failure.
std::atomic<int> g_fail_allocs{0};

cudaError_t dev_malloc(void** p, size_t bytes) {
  int n = g_fail_allocs.load();
  while (n > 0)
    if (g_fail_allocs.compare_exchange_weak(n, n - 1)) {
      *p = nullptr;
      return cudaErrorMemoryAllocation;
    }
  return cudaMalloc(p, bytes);
}

// Device memory that the current device's kernels may use as floats: where a buffer is not (host
// memory, another GPU's, not on a 4-byte boundary) the calls go through a copy instead.
bool kernel_ptr(const void* p, int dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (a.type != cudaMemoryTypeManaged && !(a.type == cudaMemoryTypeDevice && a.device == dev)) return false;
  return (reinterpret_cast<uintptr_t>(p) & 3) == 0;
}

bool is_device_ptr(const void* p) {
  if (!p) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// The side streams of a step (and the main one of its capture) and the events that tie them to the
// main stream.
struct Streams {
  cudaStream_t s[3] = {};
  cudaEvent_t ev[7] = {};
  bool create() {
    for (auto& x : s)
      if (cudaStreamCreateWithFlags(&x, cudaStreamNonBlocking) != cudaSuccess) return false;
    for (auto& x : ev)
      if (cudaEventCreateWithFlags(&x, cudaEventDisableTiming) != cudaSuccess) return false;
    return true;
  }
  void destroy() {
    for (auto& x : s)
      if (x) cudaStreamDestroy(x);
    for (auto& x : ev)
      if (x) cudaEventDestroy(x);
  }
};

}  // namespace

// --------------------------------------------------------------------------------- context

struct pdg_ctx {
  pdg_config cfg{};
  int dev = 0, sms = 1;
  int V = 0, E = 0, max_pts = 0, Qmax = 0;
  bool in_frame = false;
  int steps_in_frame = 0;
  std::string err;
  char* arena = nullptr;
  size_t arena_bytes = 0;
  Job h{};                 // host mirror of the device job struct
  Job* dJ = nullptr;       // device job struct (inside the arena)
  Plan* dplan = nullptr;   // device plan holding only this job
  Job* op_job = nullptr;   // scratch job / plan for single-level operations
  Plan* op_plan = nullptr;
  int* dflag = nullptr;
  float4* mesh = nullptr;  // [7][V]: h, r, d0, d1, preconditioned gradient, Adam m, Adam v
  int* nbr = nullptr;      // [2E] neighbours of each vertex, v2e_ptr's ranges
  float2* coef = nullptr;  // [MESH_ITERS_MAX] constants of the solves
  unsigned* bar = nullptr; // grid barrier of the solves, and their error flag
  int max_degree = 0;      // largest vertex degree of the mesh (bounds the Laplacian's spectrum)
  int mesh_wait = MESH_WAIT;  // looks at a barrier of the solves before they give up
  int mesh_refuse = 0;        // cooperative launches of the solves still to be taken as refused
  bool mesh_valid = false; // a template-mesh fit has run (PDG_BUF_MESH_* readable)
  float* stage = nullptr;  // [stage_pts][3] staging of host inputs
  int stage_pts = 0;
  Shape shape;  // of its step at capacity
  Streams cap;  // of the capture
  cudaGraphExec_t gexec = nullptr;
  int graph_kernels = 0;   // kernel nodes of gexec
  bool plan_stale = true;  // dplan's item prefixes predate the current frame
  unsigned long long frame_gen = 0;  // frames begun (a batch recomputes its plan when one changes)
  std::vector<int> v2e_ptr, v2e;

  pdg_status fail(pdg_status s, const std::string& m) {
    err = m;
    return s;
  }
  pdg_status cuda(cudaError_t e, const char* what) {
    if (e == cudaSuccess) return PDG_OK;
    err = std::string(what) + ": " + cudaGetErrorString(e);
    return PDG_ERR_CUDA;
  }
};

struct pdg_batch {
  int max_jobs = 0;
  int n = 0;
  std::vector<pdg_ctx*> members;
  Plan* dplan = nullptr;
  Plan* hplan = nullptr;  // pinned host copy
  std::vector<unsigned long long> gens;  // members' frame_gen when dplan's prefixes were computed
  Streams cap;  // of the capture
  cudaGraphExec_t gexec = nullptr;
  Shape graph_shape;  // what gexec covers
  int captures = 0;
  bool dirty = true;  // membership changed since the last upload of the job table
  std::string err;
};

#define TRY(expr)                                  \
  do {                                             \
    pdg_status _s = (expr);                        \
    if (_s != PDG_OK) return _s;                   \
  } while (0)
#define CU(ctx, call) TRY((ctx)->cuda((call), #call))

namespace {

// sizes of every buffer of a context (used by pdg_query_bytes and pdg_create)
// Chebyshev iterations of a template-mesh solve at the largest lambda times degree (1e5): 5125
constexpr int MESH_ITERS_MAX = 5200;

struct Layout {
  size_t total = 0;
  size_t job, plan, flag, stage, op_job, op_plan;
  struct Lv {
    size_t theta, theta_t, m, v, g, tmp, zmask, piv, piv_slow, mu, tw, twm, tw4, cnt, rowptr, act_v, act_ptr, ent, n_active,
        csum;
    int cap;
  } lv[MAXL];
  size_t x, y, gfwd, gy, zq, uq, gz, acc, loss_fwd, loss_rev, loss_iso, nn_fwd, nn_rev, edge_d, edges, e_prev, v2e_ptr, v2e;
  size_t src4, tgt4, verts4;
  struct Tr {
    size_t hist, off, keys, csum, perm, pts, lbox, nbox, sbox;
    int bits;
  } tgt, mov;
  size_t xs, slot_of, gys, step, bias, loss, status, loss_part, gmax, counters;
  size_t nbr, coef, bar;
  size_t mesh;  // template-mesh fit: 7 float4 [V] arrays (solves, preconditioned gradient, Adam moments)
};

Layout make_layout(const pdg_config& c, int V, int E, int max_pts) {
  Layout L;
  Arena a;
  const int Q = V + max_pts;
  const size_t C = c.payload == PDG_PAYLOAD_CAYLEY ? 6 : 3;
  L.job = a.take<Job>(1);
  L.plan = a.take<Plan>(1);
  L.op_job = a.take<Job>(1);
  L.op_plan = a.take<Plan>(1);
  L.flag = a.take<int>(4);
  const int sp = std::max(V, max_pts);
  L.stage = a.take<float>(3 * (size_t)sp);
  for (int l = 0; l < c.n_levels; ++l) {
    const size_t n = c.res[l], n3 = n * n * n;
    auto& v = L.lv[l];
    v.cap = (int)std::min<size_t>(n3, 8 * (size_t)Q);
    v.theta = a.take<float4>(n3);
    v.theta_t = a.take<float4>(C == 6 ? n3 : 1);
    v.m = a.take<float>(C * n3);
    v.v = a.take<float>(C * n3);
    v.g = a.take<float>(C * n3);
    v.tmp = a.take<float>(C * n3);
    v.zmask = a.take<int>(n);
    v.piv = a.take<float>(tile_level(n) ? 1 : (n / 2 + 1) * n * n);
    v.piv_slow = a.take<int>(1);
    v.mu = a.take<float>(n);
    v.tw = a.take<float2>(n);
    v.twm = a.take<float2>(tile_level(n) ? n : 1);
    v.tw4 = a.take<float2>(n);
    v.cnt = a.take<int>(n3);
    v.rowptr = a.take<int>(n3 + 1);
    v.act_v = a.take<int>(v.cap);
    v.act_ptr = a.take<int>(v.cap + 1);
    v.ent = a.take<int2>(8 * (size_t)Q);
    v.n_active = a.take<int>(1);
    v.csum = a.take<unsigned long long>((n3 + 1) / SCAN_CHUNK + 2);
  }
  L.x = a.take<float4>(Q);
  L.y = a.take<float4>(Q);
  L.gfwd = a.take<float4>(Q);
  L.gy = a.take<float4>(Q);
  L.zq = a.take<float4>(C == 6 ? Q : 1);
  L.uq = a.take<float4>(C == 6 ? Q : 1);
  const int vn = (V + NODE - 1) / NODE, pn = (max_pts + NODE - 1) / NODE;
  const size_t slots = (size_t)(vn + pn) * NODE;
  L.gz = a.take<float4>(C == 6 ? slots : 1);
  L.gys = a.take<float4>(slots);
  L.acc = a.take<long long>(3 * (size_t)Q);
  L.loss_fwd = a.take<float>(Q);
  L.loss_rev = a.take<float>(2 * (size_t)max_pts);
  L.loss_iso = a.take<float>(std::max(E, 1));
  L.nn_fwd = a.take<int>(Q);
  L.nn_rev = a.take<int>(2 * (size_t)max_pts);
  L.edge_d = a.take<float4>(std::max(E, 1));
  L.edges = a.take<int2>(std::max(E, 1));
  L.e_prev = a.take<float>(std::max(E, 1));
  L.v2e_ptr = a.take<int>(V + 1);
  L.v2e = a.take<int>(std::max(2 * E, 1));
  L.src4 = a.take<float4>(max_pts);
  L.tgt4 = a.take<float4>(max_pts);
  L.verts4 = a.take<float4>(V);
  auto tree = [&](Layout::Tr& t, int sets, long count, int points, int nodes) {
    t.bits = grid_bits(count);
    const size_t cells = (size_t)sets << (3 * t.bits);
    t.hist = a.take<int>(cells);
    t.off = a.take<int>(cells + 1);
    t.keys = a.take<int>(points);
    t.csum = a.take<int>(cells / SCAN_CHUNK + 2);
    t.perm = a.take<int>((size_t)nodes * NODE);
    t.pts = a.take<float>((size_t)nodes * NODE * 3);
    t.lbox = a.take<float4>((size_t)nodes * (NODE / LEAF) * 2);
    t.nbox = a.take<float4>((size_t)nodes * 2);
    t.sbox = a.take<float4>(((size_t)nodes / 32 + 2) * 2);
  };
  tree(L.tgt, 1, max_pts, max_pts, pn);
  tree(L.mov, 2, std::max(V, max_pts), Q, vn + pn);
  L.xs = a.take<float4>(slots);
  L.slot_of = a.take<int>(Q);
  L.loss_part = a.take<float>(5 * ((Q + 2 * (size_t)max_pts + std::max(E, 1)) / LOSS_CHUNK + 2));
  L.step = a.take<int>(1);
  L.bias = a.take<float>(2);
  L.loss = a.take<double>(4);
  L.status = a.take<int>(1);
  L.gmax = a.take<unsigned>(1);
  L.counters = a.take<unsigned long long>(4);
  L.mesh = a.take<float4>(7 * (size_t)V);
  L.nbr = a.take<int>(std::max(2 * E, 1));
  L.coef = a.take<float2>(MESH_ITERS_MAX);
  L.bar = a.take<unsigned>(2);
  L.total = (a.off + 255) & ~size_t(255);
  return L;
}

const char* check_config(const pdg_config* c) {
  if (!c) return "config is NULL";
  if (c->n_levels < 1 || c->n_levels > PDG_MAX_LEVELS) return "n_levels must be in 1..8";
  for (int l = 0; l < c->n_levels; ++l)
    if (!valid_res(c->res[l])) return "each res must be 1 or 2^a 3^b in 2..256";
  if (c->payload != PDG_PAYLOAD_DISPLACEMENT && c->payload != PDG_PAYLOAD_CAYLEY) return "unknown payload";
  if (c->payload == PDG_PAYLOAD_CAYLEY)
    for (int l = 0; l < c->n_levels; ++l)
      if (tile_level(c->res[l]))
        return "the Cayley payload takes levels of 1 or a power of two up to 128 vertices per axis";
  for (int a = 0; a < 3; ++a)
    if (!(std::isfinite(c->lo[a]) && std::isfinite(c->hi[a]) && c->hi[a] > c->lo[a])) return "domain must have lo < hi";
  const float f[] = {c->alpha, c->w_chamfer_mesh, c->w_chamfer_pts, c->w_iso, c->lr0, c->lr_growth, c->lambda0,
                     c->lambda_growth, c->beta1, c->beta2, c->eps};
  for (float v : f)
    if (!std::isfinite(v) || v < 0) return "config parameters must be finite and non-negative";
  if (c->beta1 >= 1 || c->beta2 >= 1) return "beta1, beta2 must be < 1";
  return nullptr;
}

// copies `n` xyz triples (host or device) into a float4 device array
pdg_status load_points(pdg_ctx* c, const float* xyz, int n, float4* dst, cudaStream_t s, bool check) {
  if (n <= 0) return PDG_OK;
  const float* src = xyz;
  if (!is_device_ptr(xyz)) {
    if (n > c->stage_pts) return c->fail(PDG_ERR_BUDGET, "point count exceeds the context capacity");
    CU(c, cudaMemcpyAsync(c->stage, xyz, sizeof(float) * 3 * (size_t)n, cudaMemcpyHostToDevice, s));
    src = c->stage;
  }
  if (check) {
    CU(c, cudaMemsetAsync(c->dflag, 0, sizeof(int), s));
    launch_check_finite(src, 3 * n, c->dflag, s);
    int f = 0;
    CU(c, cudaMemcpyAsync(&f, c->dflag, sizeof(int), cudaMemcpyDeviceToHost, s));
    CU(c, cudaStreamSynchronize(s));
    if (f) return c->fail(PDG_ERR_INVALID, "input points contain NaN or Inf");
  }
  launch_pack4(src, dst, n, s);
  return c->cuda(cudaGetLastError(), "pack points");
}

// Copies the host mirror of the job record to the device.  The mirror does not hold what the
// plan kernel writes into the device record (each level's adjoint lanes per row), so the
// plan of the context, and of any batch holding it, is recomputed before the next step.
pdg_status upload_job(pdg_ctx* c, cudaStream_t s) {
  launch_job(c->h, c->dJ, s);
  CU(c, cudaGetLastError());
  c->plan_stale = true;
  ++c->frame_gen;
  return PDG_OK;
}

// The step as an explicit list of stages; the graph capture and the profiling path launch
// exactly the same sequence.
const char* const STAGE_NAMES[] = {"interp",       "boxes",   "nn",         "nn_rev_mesh", "nn_rev_pts", "iso_edges",
                                   "assemble",     "adjoint_rows", "adjoint", "sob_xy_fwd",  "sob_z",      "sob_xy_inv",
                                   "adam",         "sobolev_256", "loss"};
constexpr int N_STAGES = sizeof(STAGE_NAMES) / sizeof(STAGE_NAMES[0]);
enum StageIndex {
  S_INTERP = 0, S_BOXES, S_NN, S_NN_REV0, S_NN_REV1, S_ISO, S_ASSEMBLE, S_ADJOINT_ROWS, S_ADJOINT,
  S_SOB_XY_FWD, S_SOB_Z, S_SOB_XY_INV, S_ADAM, S_SOB_256, S_LOSS
};

// Stage i of a step; bump: the job_bump mode of the interpolation stage (1: optimisation
// step, 2: evaluation); count: the nearest-neighbour instances that count candidates and
// exact ties.  The plan's item prefixes must be current (refresh_plan).
void launch_stage(int i, const Plan* plan, const Shape& sh, cudaStream_t s, int bump = 1, bool count = false) {
  const bool planes = sh.w[Shape::PLANES] > 0;
  switch (i) {
    case S_INTERP: launch_interp(plan, sh.blocks(Shape::NODES), s, bump); break;
    case S_BOXES: launch_boxes(plan, sh.blocks(Shape::SUPERS), s); break;
    case S_NN: launch_nn(plan, sh.blocks(Shape::NNF), s, -1, sh.nn_sub(), count); break;
    case S_NN_REV0: launch_nn(plan, sh.blocks(Shape::NNR), s, 0, sh.nn_sub(), count); break;
    case S_NN_REV1: launch_nn(plan, sh.blocks(Shape::NNR), s, 1, sh.nn_sub(), count); break;
    case S_ISO: launch_iso_edges(plan, sh.blocks(Shape::EDGES), s); break;
    case S_ASSEMBLE: launch_assemble(plan, sh.blocks(Shape::POINTS), s); break;
    case S_ADJOINT_ROWS: launch_adjoint_rows(plan, sh.blocks(Shape::ROWS), s); break;
    case S_ADJOINT: launch_adjoint(plan, sh.blocks(Shape::ADJ), s); break;
    case S_SOB_XY_FWD:
    case S_SOB_XY_INV:
      if (planes) launch_sobolev_plane(plan, sh.blocks(Shape::PLANES), sh.nmax, s, i - S_SOB_XY_FWD, sh.ext);
      break;
    case S_SOB_Z:
      if (planes) launch_sobolev_plane(plan, sh.blocks(Shape::COLS), sh.nmax, s, i - S_SOB_XY_FWD, sh.ext);
      break;
    case S_ADAM:
      if (planes) launch_sobolev_plane(plan, sh.blocks(Shape::ADAM), sh.nmax, s, i - S_SOB_XY_FWD, sh.ext);
      break;
    case S_SOB_256:
      if (sh.nline == 0) break;
      launch_sobolev_x(plan, sh.blocks(Shape::XT), sh.nline, true, s);
      for (int p = YZ_FWD; p <= YZ_INV; ++p) launch_sobolev_yz(plan, sh.blocks(Shape::YZ), sh.nline, p, s);
      launch_sobolev_x(plan, sh.blocks(Shape::XT), sh.nline, false, s);
      break;
    case S_LOSS: launch_loss(plan, sh.blocks(Shape::LOSS), sh.blocks(Shape::JOBS), s); break;
  }
}

// One step on `main` (launched, or captured into a graph), or with eval only the loss and its
// gradients.  Branches: the searches of the moving points (in the target tree, which needs no boxes
// of this step) and the isometry beside the moving trees' upper boxes and the targets' searches, one
// per moving set; the two adjoint kernels beside each other; the loss reduction beside the adjoint
// and the preconditioner (nothing downstream reads it).  All of it ends on `main`.
void launch_step(const Plan* plan, const Shape& sh, const Streams& st, cudaStream_t main, bool count, bool eval) {
  const cudaStream_t side = st.s[1], side2 = st.s[2];
  int n_ev = 0;
  auto after = [&](cudaStream_t to, cudaStream_t from) {  // `to` goes on after what `from` holds now
    cudaEventRecord(st.ev[n_ev], from);
    cudaStreamWaitEvent(to, st.ev[n_ev++], 0);
  };
  launch_stage(S_INTERP, plan, sh, main, eval ? 2 : 1);  // starts the step of every job
  after(side, main);
  launch_stage(S_BOXES, plan, sh, side);
  after(side2, side);
  launch_stage(S_NN_REV0, plan, sh, side, 1, count);
  launch_stage(S_NN_REV1, plan, sh, side2, 1, count);
  launch_stage(S_NN, plan, sh, main, 1, count);
  launch_stage(S_ISO, plan, sh, main);
  after(main, side);
  after(main, side2);
  launch_stage(S_ASSEMBLE, plan, sh, main);
  after(side, main);
  launch_stage(S_ADJOINT_ROWS, plan, sh, side);
  launch_stage(S_ADJOINT, plan, sh, main);
  after(main, side);
  launch_stage(S_LOSS, plan, sh, side);
  if (!eval)
    for (int i = S_SOB_XY_FWD; i <= S_SOB_256; ++i) launch_stage(i, plan, sh, main);  // preconditioner, Adam
  after(main, side);
}

pdg_status capture_step(pdg_ctx* c, const Plan* plan, const Shape& sh, const Streams& st, cudaGraphExec_t* out,
                        std::string* err, int* n_kernels = nullptr) {
  const cudaStream_t cap = st.s[0];
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) {
    *err = std::string("cudaStreamBeginCapture: ") + cudaGetErrorString(e);
    return PDG_ERR_CUDA;
  }
  launch_step(plan, sh, st, cap, c && c->h.count_nn, false);  // a batch graph never counts
  e = cudaStreamEndCapture(cap, &g);
  if (e != cudaSuccess) {
    *err = std::string("cudaStreamEndCapture: ") + cudaGetErrorString(e);
    if (g) cudaGraphDestroy(g);
    return PDG_ERR_CUDA;
  }
  if (n_kernels) {  // count the kernel nodes (what one replay launches)
    size_t nn = 0;
    *n_kernels = 0;
    if (cudaGraphGetNodes(g, nullptr, &nn) == cudaSuccess && nn > 0) {
      std::vector<cudaGraphNode_t> nodes(nn);
      if (cudaGraphGetNodes(g, nodes.data(), &nn) == cudaSuccess)
        for (size_t i = 0; i < nn; ++i) {
          cudaGraphNodeType t;
          if (cudaGraphNodeGetType(nodes[i], &t) == cudaSuccess && t == cudaGraphNodeTypeKernel) ++*n_kernels;
        }
    }
  }
  e = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) {
    *err = std::string("cudaGraphInstantiate: ") + cudaGetErrorString(e);
    return PDG_ERR_CUDA;
  }
  (void)c;
  return PDG_OK;
}

}  // namespace

extern "C" {

void pdg_config_default(pdg_config* c) {
  if (!c) return;
  std::memset(c, 0, sizeof(*c));
  c->n_levels = 4;
  c->res[0] = 16;
  c->res[1] = 32;
  c->res[2] = 64;
  c->res[3] = 128;
  for (int a = 0; a < 3; ++a) {
    c->lo[a] = -1.5f;
    c->hi[a] = 1.5f;
  }
  c->alpha = 5.56f;
  c->w_chamfer_mesh = 1.f;
  c->w_chamfer_pts = 1.f;
  c->w_iso = 250.f;
  c->lr0 = 5e-3f;
  c->lr_growth = 1.1f;
  c->lambda0 = 0.25f;
  c->lambda_growth = 1.5f;
  c->beta1 = 0.9f;
  c->beta2 = 0.999f;
  c->eps = 1e-8f;
  c->precondition = 1;
  c->robust_weight_stopgrad = 0;
  c->warm_start = 0;
  c->payload = PDG_PAYLOAD_DISPLACEMENT;
}

size_t pdg_query_bytes(const pdg_config* cfg, int n_verts, int n_edges, int max_pts) {
  if (check_config(cfg) || n_verts < 1 || n_edges < 0 || max_pts < 1) return 0;
  return make_layout(*cfg, n_verts, n_edges, max_pts).total;
}

const char* pdg_status_string(pdg_status s) {
  switch (s) {
    case PDG_OK: return "ok";
    case PDG_ERR_INVALID: return "invalid argument";
    case PDG_ERR_OOM: return "out of device memory";
    case PDG_ERR_BUDGET: return "over budget or capacity";
    case PDG_ERR_CUDA: return "CUDA error";
    case PDG_ERR_NONFINITE: return "non-finite loss";
    case PDG_ERR_TIMEOUT: return "device wait timed out";
    case PDG_ERR_STATE: return "call out of order";
  }
  return "unknown status";
}

const char* pdg_last_error(const pdg_ctx* c) { return c ? c->err.c_str() : "context is NULL"; }

void pdg_destroy(pdg_ctx* c) {
  if (!c) return;
  if (c->gexec) cudaGraphExecDestroy(c->gexec);
  c->cap.destroy();
  if (c->arena) cudaFree(c->arena);
  delete c;
}

pdg_status pdg_create(const pdg_config* cfg, const float* template_xyz, int n_verts, const int32_t* edges,
                      int n_edges, const float* source_xyz, int n_src, int max_pts, void* cuda_stream,
                      pdg_ctx** out) {
  if (!out) return PDG_ERR_INVALID;
  *out = nullptr;
  if (check_config(cfg) || !template_xyz || !source_xyz || n_verts < 1 || n_src < 1 || max_pts < n_src ||
      n_edges < 0 || (n_edges > 0 && !edges))
    return PDG_ERR_INVALID;
  if ((long)n_verts + max_pts > (1L << 29) || (long)n_edges > (1L << 28)) return PDG_ERR_BUDGET;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  pdg_ctx* c = new pdg_ctx();
  c->cfg = *cfg;
  c->V = n_verts;
  c->E = n_edges;
  c->max_pts = max_pts;
  c->Qmax = n_verts + max_pts;
  auto bail = [&](pdg_status st) {
    pdg_destroy(c);
    return st;
  };
  if (cudaGetDevice(&c->dev) != cudaSuccess) return bail(PDG_ERR_CUDA);
  cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, c->dev);
  c->shape.sms = c->sms;
  c->shape.add_points(n_verts, max_pts, max_pts, n_edges);
  sobolev_x_configure();
  sobolev_yz_configure();
  sobolev_plane_configure();

  // edges to the host (validation + vertex -> edge lists)
  std::vector<int32_t> he(2 * (size_t)n_edges);
  if (n_edges) {
    if (is_device_ptr(edges)) {
      if (cudaMemcpy(he.data(), edges, he.size() * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return bail(PDG_ERR_CUDA);
    } else {
      std::memcpy(he.data(), edges, he.size() * 4);
    }
  }
  for (size_t i = 0; i < he.size(); ++i)
    if (he[i] < 0 || he[i] >= n_verts) return bail(PDG_ERR_INVALID);
  c->v2e_ptr.assign(n_verts + 1, 0);
  for (int e = 0; e < n_edges; ++e) {
    c->v2e_ptr[he[2 * e] + 1]++;
    c->v2e_ptr[he[2 * e + 1] + 1]++;
  }
  for (int v = 0; v < n_verts; ++v) {
    c->max_degree = std::max(c->max_degree, c->v2e_ptr[v + 1]);
    c->v2e_ptr[v + 1] += c->v2e_ptr[v];
  }
  c->v2e.assign(std::max(2 * n_edges, 1), 0);
  {
    std::vector<int> fill(c->v2e_ptr.begin(), c->v2e_ptr.end() - 1);
    for (int e = 0; e < n_edges; ++e) {  // ascending edge order within each vertex
      c->v2e[fill[he[2 * e]]++] = e << 1;
      c->v2e[fill[he[2 * e + 1]]++] = (e << 1) | 1;
    }
  }

  std::vector<int> nbr(c->v2e.size());
  for (size_t k = 0; k < 2 * (size_t)n_edges; ++k) nbr[k] = he[2 * (size_t)(c->v2e[k] >> 1) + (c->v2e[k] & 1 ? 0 : 1)];

  const Layout L = make_layout(*cfg, n_verts, n_edges, max_pts);
  if (dev_malloc((void**)&c->arena, L.total) != cudaSuccess) {
    cudaGetLastError();
    c->arena = nullptr;
    return bail(PDG_ERR_OOM);
  }
  c->arena_bytes = L.total;
  if (cudaMemsetAsync(c->arena, 0, L.total, s) != cudaSuccess) return bail(PDG_ERR_CUDA);
  char* A = c->arena;
  auto P = [&](size_t off) { return (void*)(A + off); };
  Job& J = c->h;
  std::memset(&J, 0, sizeof(J));
  J.L = cfg->n_levels;
  J.C = cfg->payload == PDG_PAYLOAD_CAYLEY ? 6 : 3;
  for (int a = 0; a < 3; ++a) {
    J.lo[a] = cfg->lo[a];
    J.hi[a] = cfg->hi[a];
  }
  J.alpha = cfg->alpha;
  J.w_mesh = cfg->w_chamfer_mesh;
  J.w_pts = cfg->w_chamfer_pts;
  J.w_iso = cfg->w_iso;
  J.stopgrad = cfg->robust_weight_stopgrad ? 1 : 0;
  J.precondition = cfg->precondition ? 1 : 0;
  J.beta1 = cfg->beta1;
  J.beta2 = cfg->beta2;
  J.eps = cfg->eps;
  J.V = n_verts;
  J.N = n_src;
  J.M = 1;
  J.E = n_edges;
  J.Q = n_verts + n_src;
  J.max_pts = max_pts;
  c->dJ = (Job*)P(L.job);
  c->dplan = (Plan*)P(L.plan);
  c->op_job = (Job*)P(L.op_job);
  c->op_plan = (Plan*)P(L.op_plan);
  c->dflag = (int*)P(L.flag);
  c->mesh = (float4*)P(L.mesh);
  c->nbr = (int*)P(L.nbr);
  c->coef = (float2*)P(L.coef);
  c->bar = (unsigned*)P(L.bar);
  c->stage = (float*)P(L.stage);
  c->stage_pts = std::max(n_verts, max_pts);
  std::vector<float> mu;
  std::vector<float2> tw, tw4, twm;
  for (int l = 0; l < J.L; ++l) {
    Level& lv = J.lev[l];
    const auto& o = L.lv[l];
    const int n = cfg->res[l];
    lv.n = n;
    lv.n3 = n * n * n;
    lv.lr = (float)(cfg->lr0 * std::pow((double)cfg->lr_growth, l) * (cfg->precondition ? 1.0 : 0.1));
    lv.lam = (float)(cfg->lambda0 * std::pow((double)cfg->lambda_growth, l));
    for (int a = 0; a < 3; ++a) {
      const double sc = (n - 1) / ((double)cfg->hi[a] - (double)cfg->lo[a]);
      lv.sc_hi[a] = (float)sc;
      lv.sc_lo[a] = (float)(sc - (double)lv.sc_hi[a]);
    }
    lv.theta = (float4*)P(o.theta);
    lv.theta_t = J.C == 6 ? (float4*)P(o.theta_t) : nullptr;
    lv.m = (float*)P(o.m);
    lv.v = (float*)P(o.v);
    lv.g = (float*)P(o.g);
    lv.tmp = (float*)P(o.tmp);
    lv.zmask = (int*)P(o.zmask);
    lv.piv = (float*)P(o.piv);
    lv.piv_slow = (int*)P(o.piv_slow);
    lv.mu = (float*)P(o.mu);
    lv.tw = (float2*)P(o.tw);
    lv.twm = (float2*)P(o.twm);
    lv.tw4 = (float2*)P(o.tw4);
    lv.cnt = (int*)P(o.cnt);
    lv.rowptr = (int*)P(o.rowptr);
    lv.act_v = (int*)P(o.act_v);
    lv.act_ptr = (int*)P(o.act_ptr);
    lv.ent = (int2*)P(o.ent);
    lv.n_active = (int*)P(o.n_active);
    lv.csum = (unsigned long long*)P(o.csum);
    c->shape.add_level(n, J.C, c->Qmax);
    mu.resize(n);
    tw.resize(n);
    tw4.resize(n);
    for (int k = 0; k < n; ++k) {
      const double sk = std::sin(PI * k / (2.0 * n));
      mu[k] = (float)(4.0 * sk * sk);
      tw4[k] = make_float2((float)std::cos(PI * k / (2.0 * n)), (float)-std::sin(PI * k / (2.0 * n)));
    }
    for (int k = 0; k < n; ++k)
      tw[k] = make_float2((float)std::cos(2 * PI * k / n), (float)-std::sin(2 * PI * k / n));
    // pageable sources are staged before the call returns, so the vectors may be reused
    if (cudaMemcpyAsync(lv.mu, mu.data(), n * sizeof(float), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(lv.tw, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(lv.tw4, tw4.data(), n * sizeof(float2), cudaMemcpyHostToDevice, s) != cudaSuccess)
      return bail(PDG_ERR_CUDA);
    if (tile_level(n)) {
      const int n1 = line_n1(n);
      twm.resize(n);
      for (int i = 0; i < n; ++i) twm[i] = tw[(i / n1) * (i % n1)];
      if (cudaMemcpyAsync(lv.twm, twm.data(), n * sizeof(float2), cudaMemcpyHostToDevice, s) != cudaSuccess)
        return bail(PDG_ERR_CUDA);
    }
    if (!tile_level(n)) launch_sobz_pivots(lv.piv, lv.piv_slow, lv.mu, n, lv.lam, s);
  }
  J.x = (float4*)P(L.x);
  J.y = (float4*)P(L.y);
  J.gfwd = (float4*)P(L.gfwd);
  J.gy = (float4*)P(L.gy);
  J.zq = J.C == 6 ? (float4*)P(L.zq) : nullptr;
  J.uq = J.C == 6 ? (float4*)P(L.uq) : nullptr;
  J.gz = J.C == 6 ? (float4*)P(L.gz) : nullptr;
  J.acc = (long long*)P(L.acc);
  J.loss_fwd = (float*)P(L.loss_fwd);
  J.loss_rev = (float*)P(L.loss_rev);
  J.loss_iso = (float*)P(L.loss_iso);
  J.nn_fwd = (int*)P(L.nn_fwd);
  J.nn_rev = (int*)P(L.nn_rev);
  J.edge_d = (float4*)P(L.edge_d);
  J.edges = (const int2*)P(L.edges);
  J.e_prev = (float*)P(L.e_prev);
  J.v2e_ptr = (const int*)P(L.v2e_ptr);
  J.v2e = (const int*)P(L.v2e);
  J.src4 = (float4*)P(L.src4);
  J.tgt4 = (float4*)P(L.tgt4);
  J.verts4 = (float4*)P(L.verts4);
  auto tree_init = [&](Tree& t, const Layout::Tr& o) {
    t.bits = o.bits;
    for (int a = 0; a < 3; ++a) {
      t.lo[a] = cfg->lo[a];
      t.inv_h[a] = (float)((1 << o.bits) / ((double)cfg->hi[a] - cfg->lo[a]));
    }
    t.hist = (int*)P(o.hist);
    t.off = (int*)P(o.off);
    t.keys = (int*)P(o.keys);
    t.csum = (int*)P(o.csum);
    t.perm = (int*)P(o.perm);
    t.pts = (float*)P(o.pts);
    t.lbox = (float4*)P(o.lbox);
    t.nbox = (float4*)P(o.nbox);
    t.sbox = (float4*)P(o.sbox);
  };
  tree_init(J.tgt, L.tgt);
  tree_init(J.mov, L.mov);
  J.xs = (float4*)P(L.xs);
  J.slot_of = (int*)P(L.slot_of);
  J.gys = (float4*)P(L.gys);
  J.loss_part = (float*)P(L.loss_part);
  J.step = (int*)P(L.step);
  J.bias = (float*)P(L.bias);
  J.loss = (double*)P(L.loss);
  J.status = (int*)P(L.status);
  J.gmax = (unsigned*)P(L.gmax);
  J.counters = (unsigned long long*)P(L.counters);

  if (n_edges) {
    if (cudaMemcpyAsync((void*)J.edges, he.data(), he.size() * 4, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync((void*)J.v2e, c->v2e.data(), c->v2e.size() * 4, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(c->nbr, nbr.data(), nbr.size() * 4, cudaMemcpyHostToDevice, s) != cudaSuccess)
      return bail(PDG_ERR_CUDA);
  }
  if (cudaMemcpyAsync((void*)J.v2e_ptr, c->v2e_ptr.data(), c->v2e_ptr.size() * 4, cudaMemcpyHostToDevice, s) !=
      cudaSuccess)
    return bail(PDG_ERR_CUDA);
  if (load_points(c, template_xyz, n_verts, J.verts4, s, true) != PDG_OK) {
    const pdg_status st = c->err.find("NaN") != std::string::npos ? PDG_ERR_INVALID : PDG_ERR_CUDA;
    return bail(st);
  }
  if (load_points(c, source_xyz, n_src, J.src4, s, true) != PDG_OK) {
    const pdg_status st = c->err.find("NaN") != std::string::npos ? PDG_ERR_INVALID : PDG_ERR_CUDA;
    return bail(st);
  }
  if (upload_job(c, s) != PDG_OK) return bail(PDG_ERR_CUDA);
  {
    Plan hp;
    std::memset(&hp, 0, sizeof(hp));
    hp.n_jobs = 1;
    hp.jobs[0] = c->dJ;
    if (cudaMemcpyAsync(c->dplan, &hp, sizeof(Plan), cudaMemcpyHostToDevice, s) != cudaSuccess)
      return bail(PDG_ERR_CUDA);
  }
  if (!c->cap.create())
    return bail(PDG_ERR_CUDA);
  if (cudaStreamSynchronize(s) != cudaSuccess) return bail(PDG_ERR_CUDA);
  *out = c;
  return PDG_OK;
}

pdg_status pdg_set_debug(pdg_ctx* c, int flags) {
  if (!c || (flags & ~(PDG_DEBUG_KEEP_PGRAD | PDG_DEBUG_COUNT_NN))) return PDG_ERR_INVALID;
  c->h.keep_pgrad = (flags & PDG_DEBUG_KEEP_PGRAD) ? 1 : 0;
  const int count = (flags & PDG_DEBUG_COUNT_NN) ? 1 : 0;
  if (count != c->h.count_nn && c->gexec) {  // the step graph holds the other NN instances
    if (cudaDeviceSynchronize() != cudaSuccess) return PDG_ERR_CUDA;
    cudaGraphExecDestroy(c->gexec);
    c->gexec = nullptr;
  }
  c->h.count_nn = count;
  return upload_job(c, 0) == PDG_OK ? c->cuda(cudaDeviceSynchronize(), "set_debug") : PDG_ERR_CUDA;
}

// Recomputes the context's plan prefixes (stream-ordered) if a frame began since the last time.
pdg_status refresh_plan(pdg_ctx* c, cudaStream_t s) {
  if (!c->plan_stale) return PDG_OK;
  launch_plan(c->dplan, s);
  CU(c, cudaGetLastError());
  c->plan_stale = false;
  return PDG_OK;
}

pdg_status pdg_begin_frame(pdg_ctx* c, const float* target_xyz, int n_tgt, void* cuda_stream) {
  if (!c) return PDG_ERR_INVALID;
  if (c->in_frame) return c->fail(PDG_ERR_STATE, "a frame is already open");
  if (!target_xyz || n_tgt < 1) return c->fail(PDG_ERR_INVALID, "empty target");
  if (n_tgt > c->max_pts) return c->fail(PDG_ERR_BUDGET, "target larger than max_pts");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  Job& J = c->h;
  TRY(load_points(c, target_xyz, n_tgt, J.tgt4, s, true));
  J.M = n_tgt;
  J.Q = J.V + J.N;
  TRY(upload_job(c, s));
  launch_frame_points(c->dJ, J.Q, J.E, s);
  // A level's theta, theta_t, m, v and g follow one another in the arena (see make_layout), as do the
  // step count, bias corrections, losses and status: one clearing each.
  for (int l = 0; l < J.L; ++l) {
    const Level& lv = J.lev[l];
    char* from = c->cfg.warm_start ? (char*)lv.m : (char*)lv.theta;
    CU(c, cudaMemsetAsync(from, 0, (char*)(lv.g + (size_t)J.C * lv.n3) - from, s));
  }
  CU(c, cudaMemsetAsync(J.step, 0, (char*)(J.status + 1) - (char*)J.step, s));
  launch_tree_build(c->dJ, J, s);
  launch_nn_seed(c->dJ, J, s);
  launch_csr_build(c->dJ, J, s);
  CU(c, cudaGetLastError());
  c->in_frame = true;
  c->mesh_valid = false;  // the step overwrites the mesh fit's gradient
  c->steps_in_frame = 0;
  c->plan_stale = true;
  ++c->frame_gen;
  return PDG_OK;
}

pdg_status pdg_step(pdg_ctx* c, int n_steps, void* cuda_stream) {
  if (!c) return PDG_ERR_INVALID;
  if (!c->in_frame) return c->fail(PDG_ERR_STATE, "pdg_step outside a frame");
  if (n_steps < 0) return c->fail(PDG_ERR_INVALID, "negative step count");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  if (!c->gexec) {
    // the captured launches must not start before this stream's pending set-up
    CU(c, cudaStreamSynchronize(s));
    TRY(capture_step(c, c->dplan, c->shape, c->cap, &c->gexec, &c->err, &c->graph_kernels));
  }
  TRY(refresh_plan(c, s));
  for (int i = 0; i < n_steps; ++i) CU(c, cudaGraphLaunch(c->gexec, s));
  c->steps_in_frame += n_steps;
  return PDG_OK;
}

int pdg_profile_stages(void) { return N_STAGES; }

const char* pdg_profile_stage_name(int i) { return (i >= 0 && i < N_STAGES) ? STAGE_NAMES[i] : ""; }

pdg_status pdg_step_kernel_count(const pdg_ctx* c, int* out) {
  if (!c || !out) return PDG_ERR_INVALID;
  *out = c->gexec ? c->graph_kernels : 0;
  return PDG_OK;
}

pdg_status pdg_profile_step(pdg_ctx* c, int n_steps, double* stage_ms, void* cuda_stream) {
  if (!c || !stage_ms || n_steps < 0) return PDG_ERR_INVALID;
  if (!c->in_frame) return c->fail(PDG_ERR_STATE, "pdg_profile_step outside a frame");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  cudaEvent_t ev[N_STAGES + 1];
  for (auto& e : ev) CU(c, cudaEventCreate(&e));
  for (int i = 0; i < N_STAGES; ++i) stage_ms[i] = 0.0;
  pdg_status st = refresh_plan(c, s);
  for (int k = 0; k < n_steps && st == PDG_OK; ++k) {
    for (int i = 0; i < N_STAGES; ++i) {
      cudaEventRecord(ev[i], s);
      launch_stage(i, c->dplan, c->shape, s, 1, c->h.count_nn != 0);
    }
    cudaEventRecord(ev[N_STAGES], s);
    st = c->cuda(cudaEventSynchronize(ev[N_STAGES]), "profile step");
    for (int i = 0; i < N_STAGES && st == PDG_OK; ++i) {
      float ms = 0.f;
      cudaEventElapsedTime(&ms, ev[i], ev[i + 1]);
      stage_ms[i] += ms;
    }
  }
  for (auto& e : ev) cudaEventDestroy(e);
  c->steps_in_frame += n_steps;
  return st;
}

pdg_status pdg_end_frame(pdg_ctx* c, pdg_fit_stats* stats, void* cuda_stream) {
  if (!c) return PDG_ERR_INVALID;
  if (!c->in_frame) return c->fail(PDG_ERR_STATE, "no open frame");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  Job& J = c->h;
  launch_end_frame(c->dJ, J.V, s);
  CU(c, cudaMemcpyAsync(J.src4, J.tgt4, sizeof(float4) * J.M, cudaMemcpyDeviceToDevice, s));
  double loss[4];
  int status = 0;
  unsigned long long cnt[4] = {0, 0, 0, 0};
  CU(c, cudaMemcpyAsync(loss, J.loss, sizeof(loss), cudaMemcpyDeviceToHost, s));
  CU(c, cudaMemcpyAsync(&status, J.status, sizeof(int), cudaMemcpyDeviceToHost, s));
  CU(c, cudaMemcpyAsync(cnt, J.counters, sizeof(cnt), cudaMemcpyDeviceToHost, s));
  CU(c, cudaStreamSynchronize(s));
  J.N = J.M;
  J.Q = J.V + J.N;
  c->in_frame = false;
  const pdg_status st = status ? PDG_ERR_NONFINITE : PDG_OK;
  if (stats) {
    stats->loss_total = loss[0];
    stats->cd_mesh = loss[1];
    stats->cd_pts = loss[2];
    stats->iso = loss[3];
    stats->n_steps = c->steps_in_frame;
    stats->status = st;
    stats->nn_ties = !J.count_nn ? -1 : c->steps_in_frame > 0 ? (int)std::min<unsigned long long>(cnt[CNT_NN_TIES], 0x7fffffff) : 0;
  }
  if (st != PDG_OK) c->err = "a loss became NaN or Inf during the frame";
  return st;
}

pdg_status pdg_fit_frame(pdg_ctx* c, const float* target_xyz, int n_tgt, int n_steps, pdg_fit_stats* stats,
                         void* cuda_stream) {
  TRY(pdg_begin_frame(c, target_xyz, n_tgt, cuda_stream));
  const pdg_status st = pdg_step(c, n_steps, cuda_stream);
  if (st != PDG_OK) {
    c->in_frame = false;
    return st;
  }
  return pdg_end_frame(c, stats, cuda_stream);
}

pdg_status pdg_deform(pdg_ctx* c, const float* xyz, int n, float* out, void* cuda_stream) {
  if (!c) return PDG_ERR_INVALID;
  if (n < 0 || (n > 0 && (!xyz || !out))) return c->fail(PDG_ERR_INVALID, "bad deform arguments");
  if (n == 0) return PDG_OK;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const bool din = is_device_ptr(xyz), dout = is_device_ptr(out);
  if (din && dout) {
    launch_deform(c->dJ, xyz, out, n, s);
    return c->cuda(cudaGetLastError(), "deform");
  }
  // host buffers go through the context's staging area in chunks (no allocation): the first
  // half of the area holds the chunk's input, the second its output
  const int chunk = std::max(1, c->stage_pts / 2);
  float* sin_ = c->stage;
  float* sout = c->stage + 3 * (size_t)chunk;
  for (int b = 0; b < n; b += chunk) {
    const int m = std::min(chunk, n - b);
    const size_t bytes = sizeof(float) * 3 * (size_t)m;
    const float* in = xyz + 3 * (size_t)b;
    float* o = out + 3 * (size_t)b;
    if (!din) {
      CU(c, cudaMemcpyAsync(sin_, in, bytes, cudaMemcpyHostToDevice, s));
      in = sin_;
    }
    launch_deform(c->dJ, in, dout ? o : sout, m, s);
    if (!dout) CU(c, cudaMemcpyAsync(o, sout, bytes, cudaMemcpyDeviceToHost, s));
    // the next chunk overwrites the staging area: wait until this one has left it
    CU(c, cudaStreamSynchronize(s));
  }
  return c->cuda(cudaGetLastError(), "deform");
}

// copies `bytes` from a device buffer to `out` (host or device), synchronising for host
static pdg_status copy_out(pdg_ctx* c, void* out, const void* dsrc, size_t bytes, cudaStream_t s) {
  if (is_device_ptr(out)) {
    CU(c, cudaMemcpyAsync(out, dsrc, bytes, cudaMemcpyDeviceToDevice, s));
  } else {
    CU(c, cudaMemcpyAsync(out, dsrc, bytes, cudaMemcpyDeviceToHost, s));
    CU(c, cudaStreamSynchronize(s));
  }
  return PDG_OK;
}

pdg_status pdg_get_vertices(pdg_ctx* c, float* out, void* cuda_stream) {
  if (!c || !out) return PDG_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const size_t bytes = sizeof(float) * 3 * (size_t)c->V;
  if (is_device_ptr(out)) {
    launch_unpack4(c->h.verts4, out, c->V, s);
    return c->cuda(cudaGetLastError(), "get_vertices");
  }
  // through the staging area (it holds max(V, max_pts) points): no allocation
  launch_unpack4(c->h.verts4, c->stage, c->V, s);
  return copy_out(c, out, c->stage, bytes, s);
}

pdg_status pdg_read(pdg_ctx* c, int which, int level, void* out, size_t out_bytes, void* cuda_stream) {
  if (!c || !out) return PDG_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const Job& J = c->h;
  const bool per_level = which == PDG_BUF_THETA || which == PDG_BUF_GRAD || which == PDG_BUF_PGRAD;
  if (per_level && (level < 0 || level >= J.L)) return c->fail(PDG_ERR_INVALID, "bad level");
  size_t need = 0;
  switch (which) {
    case PDG_BUF_THETA:
    case PDG_BUF_GRAD:
    case PDG_BUF_PGRAD: need = sizeof(float) * J.C * (size_t)J.lev[level].n3; break;
    case PDG_BUF_Y:
    case PDG_BUF_POINT_GRAD: need = sizeof(float) * 3 * (size_t)J.Q; break;
    case PDG_BUF_NN_FWD: need = sizeof(int) * (size_t)J.Q; break;
    case PDG_BUF_NN_REV: need = sizeof(int) * 2 * (size_t)J.M; break;
    case PDG_BUF_LOSS: need = 4 * sizeof(double); break;
    case PDG_BUF_SOURCE: need = sizeof(float) * 3 * (size_t)J.N; break;
    case PDG_BUF_COUNTERS: need = 4 * sizeof(unsigned long long); break;
    case PDG_BUF_MESH_GRAD:
    case PDG_BUF_MESH_PGRAD:
      if (!c->mesh_valid) return c->fail(PDG_ERR_STATE, "no template-mesh fit has run");
      need = sizeof(float) * 3 * (size_t)c->V;
      break;
    default: return c->fail(PDG_ERR_INVALID, "unknown buffer");
  }
  if (out_bytes < need) return c->fail(PDG_ERR_INVALID, "output buffer too small");
  if (which == PDG_BUF_PGRAD && !J.keep_pgrad) return c->fail(PDG_ERR_STATE, "call pdg_set_debug(ctx, 1) first");
  if (which == PDG_BUF_LOSS) return copy_out(c, out, J.loss, need, s);
  if (which == PDG_BUF_NN_FWD) return copy_out(c, out, J.nn_fwd, need, s);
  if (which == PDG_BUF_NN_REV) return copy_out(c, out, J.nn_rev, need, s);
  if (which == PDG_BUF_COUNTERS) return copy_out(c, out, J.counters, need, s);
  // straight into a device buffer; a stream-ordered allocation would be given back to the system at the
  // next synchronisation and cost about 200 us each time
  const bool direct = kernel_ptr(out, c->dev);
  float* tmp = static_cast<float*>(out);
  if (!direct) CU(c, cudaMallocAsync((void**)&tmp, need, s));
  switch (which) {
    case PDG_BUF_THETA:
      launch_unpack_theta(J.lev[level].theta, J.lev[level].theta_t, tmp, J.lev[level].n3, J.C, s);
      break;
    case PDG_BUF_GRAD: launch_soa_to_aos(J.lev[level].g, tmp, J.lev[level].n3, s, J.C); break;
    case PDG_BUF_PGRAD:  // without the preconditioner Adam takes the raw gradient
      launch_soa_to_aos(J.precondition ? J.lev[level].tmp : J.lev[level].g, tmp, J.lev[level].n3, s, J.C);
      break;
    case PDG_BUF_Y: launch_unpack4(J.y, tmp, J.Q, s); break;
    case PDG_BUF_POINT_GRAD: launch_unpack4(J.gy, tmp, J.Q, s); break;
    case PDG_BUF_SOURCE: launch_unpack4(J.src4, tmp, J.N, s); break;
    case PDG_BUF_MESH_GRAD: launch_unpack4(J.gy, tmp, c->V, s); break;
    case PDG_BUF_MESH_PGRAD: launch_unpack4(c->mesh + 4 * (size_t)c->V, tmp, c->V, s); break;
  }
  if (direct) return c->cuda(cudaGetLastError(), "read");
  const pdg_status st = copy_out(c, out, tmp, need, s);
  cudaFreeAsync(tmp, s);
  return st;
}

pdg_status pdg_write_theta(pdg_ctx* c, int level, const float* theta, void* cuda_stream) {
  if (!c || !theta) return PDG_ERR_INVALID;
  if (level < 0 || level >= c->h.L) return c->fail(PDG_ERR_INVALID, "bad level");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const Level& lv = c->h.lev[level];
  const float* src = theta;
  float* tmp = nullptr;
  const int C = c->h.C;
  const size_t bytes = sizeof(float) * C * (size_t)lv.n3;
  if (!is_device_ptr(theta)) {
    CU(c, cudaMallocAsync((void**)&tmp, bytes, s));
    CU(c, cudaMemcpyAsync(tmp, theta, bytes, cudaMemcpyHostToDevice, s));
    src = tmp;
  }
  launch_pack_theta(src, lv.theta, lv.theta_t, lv.m, lv.v, lv.n3, C, s);
  if (tmp) {
    CU(c, cudaFreeAsync(tmp, s));
    CU(c, cudaStreamSynchronize(s));
  }
  return c->cuda(cudaGetLastError(), "write_theta");
}

pdg_status pdg_eval(pdg_ctx* c, double* loss, void* cuda_stream) {
  if (!c) return PDG_ERR_INVALID;
  if (!c->in_frame) return c->fail(PDG_ERR_STATE, "pdg_eval outside a frame");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  TRY(refresh_plan(c, s));
  launch_step(c->dplan, c->shape, c->cap, s, c->h.count_nn != 0, true);  // no preconditioner, no Adam, no step count
  CU(c, cudaGetLastError());
  if (loss) {
    CU(c, cudaMemcpyAsync(loss, c->h.loss, 4 * sizeof(double), cudaMemcpyDeviceToHost, s));
    CU(c, cudaStreamSynchronize(s));
  }
  return PDG_OK;
}

pdg_status pdg_precondition(pdg_ctx* c, int level, const float* g, float* out, void* cuda_stream) {
  if (!c || !g || !out) return PDG_ERR_INVALID;
  if (c->in_frame) return c->fail(PDG_ERR_STATE, "pdg_precondition only between frames");
  if (level < 0 || level >= c->h.L) return c->fail(PDG_ERR_INVALID, "bad level");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const Level& lv = c->h.lev[level];
  const size_t bytes = sizeof(float) * 3 * (size_t)lv.n3;
  // device buffers are read and written in place (every read of g precedes the first write of out)
  const bool direct_g = kernel_ptr(g, c->dev), direct_out = kernel_ptr(out, c->dev);
  float* tmp = nullptr;
  if (!direct_g || !direct_out) CU(c, cudaMallocAsync((void**)&tmp, bytes, s));
  if (!direct_g) CU(c, cudaMemcpyAsync(tmp, g, bytes, is_device_ptr(g) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
  const float* gin = direct_g ? g : tmp;
  float* gout = direct_out ? out : tmp;
  const bool line = line_size(lv.n) > 0;
  // a one-level copy of the job, for the passes without Adam
  Job oj = c->h;
  oj.L = 1;
  oj.C = 3;  // the entry point preconditions 3 channels whatever the payload
  oj.lev[0] = lv;
  oj.lev[0].zmask = nullptr;  // a caller's gradient may be non-zero on any plane
  oj.precondition = 1;
  oj.ext_in = gin;  // the passes read and write [n^3][3] themselves
  oj.ext_out = gout;
  launch_op_plan(oj, c->op_job, c->op_plan, s);
  Shape sh;
  sh.sms = c->sms;
  sh.add_level(lv.n, 3, 0);
  sh.ext = true;
  if (line) launch_stage(S_SOB_256, c->op_plan, sh, s);
  else
    for (int i = S_SOB_XY_FWD; i <= S_SOB_XY_INV; ++i) launch_stage(i, c->op_plan, sh, s);
  CU(c, cudaGetLastError());
  const pdg_status st = direct_out ? PDG_OK : copy_out(c, out, tmp, bytes, s);
  if (tmp) cudaFreeAsync(tmp, s);
  CU(c, cudaStreamSynchronize(s));
  return st;
}

// ------------------------------------------------------------------------------ template-mesh fit

pdg_status pdg_fit_mesh(pdg_ctx* c, const float* p0_xyz, int n_p0, int n_steps, float lambda, float lr,
                        pdg_fit_stats* stats, void* cuda_stream) {
  if (!c) return PDG_ERR_INVALID;
  if (c->in_frame) return c->fail(PDG_ERR_STATE, "pdg_fit_mesh only between frames");
  if (!p0_xyz || n_p0 < 1 || n_steps < 0 || !(lambda >= 0.f) || !(lambda < 1e30f) || !(lr >= 0.f) || !(lr < 1e30f))
    return c->fail(PDG_ERR_INVALID, "bad mesh-fit arguments");
  if (n_p0 > c->max_pts) return c->fail(PDG_ERR_BUDGET, "cloud larger than max_pts");
  // bounds the Chebyshev iteration count below (about 5000 per solve at the limit)
  if ((double)lambda * std::max(c->max_degree, 1) > 1e5)
    return c->fail(PDG_ERR_INVALID, "lambda times the largest vertex degree above 1e5");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  Job& J = c->h;
  const int V = c->V;
  TRY(load_points(c, p0_xyz, n_p0, J.tgt4, s, true));
  // the step's kernels on a job whose query points are the mesh vertices alone: no source set,
  // no isometry, the mesh term with weight 1; 3 channels (the grids take no part)
  Job mj = J;
  mj.N = 0;
  mj.Q = V;
  mj.M = n_p0;
  mj.E = 0;
  mj.C = 3;
  mj.w_mesh = 1.f;
  mj.w_pts = 0.f;
  mj.w_iso = 0.f;
  mj.count_nn = 0;
  launch_op_plan(mj, c->op_job, c->op_plan, s);
  float4* h = c->mesh;
  float4* r = h + V;
  float4* d0 = r + V;
  float4* d1 = d0 + V;
  float4* pg = d1 + V;
  float4* am = pg + V;
  float4* av = am + V;
  CU(c, cudaMemcpyAsync(J.x, J.verts4, sizeof(float4) * V, cudaMemcpyDeviceToDevice, s));  // X_0 being fitted
  CU(c, cudaMemsetAsync(am, 0, 2 * sizeof(float4) * (size_t)V, s));
  CU(c, cudaMemsetAsync(J.loss, 0, 4 * sizeof(double), s));
  CU(c, cudaMemsetAsync(J.status, 0, sizeof(int), s));
  launch_tree_build(c->op_job, mj, s);
  launch_nn_seed(c->op_job, mj, s);
  // Chebyshev interval: the Laplacian's eigenvalues lie in [0, 2 max degree] (Gershgorin), so
  // those of I + lambda L in [1, emax]; iterations for a relative error below 1e-7 in exact
  // arithmetic, 2 sqrt(kappa) q^k <= 1e-7 with q = (sqrt(kappa) - 1) / (sqrt(kappa) + 1)
  const double emax = 1.0 + 2.0 * lambda * std::max(c->max_degree, 1);
  const double sk = std::sqrt(emax);
  const double q = (sk - 1.0) / (sk + 1.0);
  const int iters = q > 0.0 ? (int)std::ceil(std::log(1e-7 / (2.0 * sk)) / std::log(q)) : 1;
  MeshSolve ms{};
  ms.ptr = J.v2e_ptr;
  ms.nbr = c->nbr;
  ms.b = J.gy;
  ms.h = h;
  ms.r = r;
  ms.d0 = d0;
  ms.d1 = d1;
  ms.pg = pg;
  ms.x = J.x;
  ms.m = am;
  ms.v = av;
  ms.coef = c->coef;
  ms.bar = c->bar;
  ms.err = reinterpret_cast<int*>(c->bar + 1);
  ms.wait = c->mesh_wait;
  ms.V = V;
  ms.iters = iters;
  ms.degree = c->max_degree;
  ms.lam = lambda;
  ms.lr = lr;
  ms.b1 = J.beta1;
  ms.b2 = J.beta2;
  ms.eps = J.eps;
  CU(c, cudaMemsetAsync(ms.err, 0, sizeof(int), s));
  std::vector<float2> coef;
  mesh_coef(coef, iters, (float)emax);
  CU(c, cudaMemcpyAsync(c->coef, coef.data(), sizeof(float2) * coef.size(), cudaMemcpyHostToDevice, s));
  Shape sh;
  sh.sms = c->sms;
  sh.add_points(V, 0, n_p0, 0);
  for (int k = 1; k <= n_steps; ++k) {
    launch_mesh_points(c->op_job, V, s);
    for (int i = S_BOXES; i <= S_NN_REV0; ++i) launch_stage(i, c->op_plan, sh, s);
    launch_stage(S_ASSEMBLE, c->op_plan, sh, s);
    launch_stage(S_LOSS, c->op_plan, sh, s);
    // (I + lambda L)^{-2} dL/dX by two solves, then Adam on the vertices
    ms.bias1 = (float)(1.0 / (1.0 - std::pow((double)J.beta1, k)));
    ms.ibias2 = (float)(1.0 / std::sqrt(1.0 - std::pow((double)J.beta2, k)));
    CU(c, launch_mesh_solve(ms, (float)emax, c->sms, c->mesh_refuse, s));
  }
  launch_mesh_commit(ms, J.verts4, s);
  CU(c, cudaGetLastError());
  double loss[4];
  int status = 0, gave_up = 0;
  CU(c, cudaMemcpyAsync(loss, J.loss, sizeof(loss), cudaMemcpyDeviceToHost, s));
  CU(c, cudaMemcpyAsync(&status, J.status, sizeof(int), cudaMemcpyDeviceToHost, s));
  CU(c, cudaMemcpyAsync(&gave_up, ms.err, sizeof(int), cudaMemcpyDeviceToHost, s));
  CU(c, cudaStreamSynchronize(s));
  c->mesh_valid = n_steps > 0 && !gave_up;
  c->plan_stale = true;  // the frame plan is recomputed at the next frame
  const pdg_status st = gave_up ? PDG_ERR_TIMEOUT : status ? PDG_ERR_NONFINITE : PDG_OK;
  if (stats) {
    stats->loss_total = loss[0];
    stats->cd_mesh = loss[1];
    stats->cd_pts = 0.0;
    stats->iso = 0.0;
    stats->n_steps = n_steps;
    stats->status = st;
    stats->nn_ties = -1;
  }
  if (st != PDG_OK)
    c->err = gave_up ? "a wait of the mesh solves ran out" : "a loss became NaN or Inf during the mesh fit";
  return st;
}

// ------------------------------------------------------------------------------ batching

pdg_status pdg_debug_mesh_wait(pdg_ctx* c, int looks) {
  if (!c || looks < 0) return PDG_ERR_INVALID;
  c->mesh_wait = looks ? looks : MESH_WAIT;
  return PDG_OK;
}

pdg_status pdg_debug_mesh_refuse(pdg_ctx* c, int n) {
  if (!c) return PDG_ERR_INVALID;
  c->mesh_refuse = std::max(n, 0);
  return PDG_OK;
}

void pdg_debug_fail_allocations(int n) { g_fail_allocs.store(n > 0 ? n : 0); }

pdg_status pdg_batch_create(int max_jobs, pdg_batch** out) {
  if (!out || max_jobs < 1 || max_jobs > MAXJ) return PDG_ERR_INVALID;
  pdg_batch* b = new pdg_batch();
  b->max_jobs = max_jobs;
  if (dev_malloc((void**)&b->dplan, sizeof(Plan)) != cudaSuccess || cudaMallocHost(&b->hplan, sizeof(Plan)) != cudaSuccess ||
      !b->cap.create()) {
    cudaGetLastError();
    pdg_batch_destroy(b);
    return PDG_ERR_OOM;
  }
  std::memset(b->hplan, 0, sizeof(Plan));
  *out = b;
  return PDG_OK;
}

void pdg_batch_destroy(pdg_batch* b) {
  if (!b) return;
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
  b->cap.destroy();
  if (b->dplan) cudaFree(b->dplan);
  if (b->hplan) cudaFreeHost(b->hplan);
  delete b;
}

pdg_status pdg_batch_set(pdg_batch* b, pdg_ctx* const* ctxs, int n_jobs) {
  if (!b || n_jobs < 0 || n_jobs > b->max_jobs || (n_jobs && !ctxs)) return PDG_ERR_INVALID;
  for (int i = 0; i < n_jobs; ++i) {
    if (!ctxs[i]) return PDG_ERR_INVALID;
    if (!ctxs[i]->in_frame) {
      b->err = "batch member outside a frame";
      return PDG_ERR_STATE;
    }
    for (int k = 0; k < i; ++k)
      if (ctxs[k] == ctxs[i]) return PDG_ERR_INVALID;
  }
  b->members.assign(ctxs, ctxs + n_jobs);
  b->n = n_jobs;
  b->dirty = true;
  return PDG_OK;
}

pdg_status pdg_batch_step(pdg_batch* b, int n_steps, void* cuda_stream) {
  if (!b || n_steps < 0) return PDG_ERR_INVALID;
  if (b->n == 0 || n_steps == 0) return PDG_OK;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  Shape sh;
  for (auto* c : b->members) {
    if (!c->in_frame) {
      b->err = "batch member outside a frame";
      return PDG_ERR_STATE;
    }
    sh.add(c->shape);
  }
  if (b->dirty) {
    // publish the membership (stream-ordered; the pinned host copy is rewritten only after
    // the previous upload completed)
    if (cudaStreamSynchronize(s) != cudaSuccess) return PDG_ERR_CUDA;
    std::memset(b->hplan, 0, sizeof(Plan));
    b->hplan->n_jobs = b->n;
    for (int i = 0; i < b->n; ++i) b->hplan->jobs[i] = b->members[i]->dJ;
    if (cudaMemcpyAsync(b->dplan, b->hplan, sizeof(Plan), cudaMemcpyHostToDevice, s) != cudaSuccess)
      return PDG_ERR_CUDA;
    b->dirty = false;
    b->gens.clear();
  }
  // item prefixes: recomputed when the membership changed or a member began a frame
  bool stale = b->gens.size() != b->members.size();
  for (size_t i = 0; i < b->members.size() && !stale; ++i) stale = b->gens[i] != b->members[i]->frame_gen;
  if (stale) {
    launch_plan(b->dplan, s);
    if (cudaGetLastError() != cudaSuccess) return PDG_ERR_CUDA;
    b->gens.resize(b->members.size());
    for (size_t i = 0; i < b->members.size(); ++i) b->gens[i] = b->members[i]->frame_gen;
  }
  // the graph is captured for the largest of every quantity so far: again only when that grows past
  // what its launches have
  Shape need = b->graph_shape;
  need.cover(sh);
  if (!b->gexec || !need.same_launches(b->graph_shape)) {
    if (b->gexec) cudaGraphExecDestroy(b->gexec);
    b->gexec = nullptr;
    if (cudaStreamSynchronize(s) != cudaSuccess) return PDG_ERR_CUDA;
    const pdg_status st = capture_step(nullptr, b->dplan, need, b->cap, &b->gexec, &b->err);
    if (st != PDG_OK) return st;
    ++b->captures;
  }
  b->graph_shape = need;
  for (int i = 0; i < n_steps; ++i)
    if (cudaGraphLaunch(b->gexec, s) != cudaSuccess) return PDG_ERR_CUDA;
  for (auto* c : b->members) c->steps_in_frame += n_steps;
  return PDG_OK;
}

pdg_status pdg_batch_graph_captures(const pdg_batch* b, int* out) {
  if (!b || !out) return PDG_ERR_INVALID;
  *out = b->captures;
  return PDG_OK;
}

// ------------------------------------------------------------------------------ state

namespace {
struct StateHeader {
  char magic[8];
  int version, V, N, L, res[PDG_MAX_LEVELS], C;
};
}  // namespace

size_t pdg_state_bytes(const pdg_ctx* c) {
  if (!c) return 0;
  size_t b = sizeof(StateHeader) + sizeof(float4) * (size_t)c->V + sizeof(float4) * (size_t)c->max_pts;
  for (int l = 0; l < c->h.L; ++l) b += sizeof(float4) * (size_t)c->h.lev[l].n3 * (c->h.C / 3);
  return b;
}

pdg_status pdg_save_state(pdg_ctx* c, void* host_buf, size_t n, void* cuda_stream) {
  if (!c || !host_buf) return PDG_ERR_INVALID;
  if (c->in_frame) return c->fail(PDG_ERR_STATE, "save only between frames");
  if (n < pdg_state_bytes(c)) return c->fail(PDG_ERR_INVALID, "state buffer too small");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  StateHeader hd{};
  std::memcpy(hd.magic, "PDGSTAT", 8);
  hd.version = 2;
  hd.V = c->V;
  hd.C = c->h.C;
  hd.N = c->h.N;
  hd.L = c->h.L;
  for (int l = 0; l < c->h.L; ++l) hd.res[l] = c->h.lev[l].n;
  char* p = (char*)host_buf;
  std::memcpy(p, &hd, sizeof(hd));
  p += sizeof(hd);
  CU(c, cudaMemcpyAsync(p, c->h.verts4, sizeof(float4) * c->V, cudaMemcpyDeviceToHost, s));
  p += sizeof(float4) * c->V;
  CU(c, cudaMemcpyAsync(p, c->h.src4, sizeof(float4) * c->max_pts, cudaMemcpyDeviceToHost, s));
  p += sizeof(float4) * c->max_pts;
  for (int l = 0; l < c->h.L; ++l) {
    CU(c, cudaMemcpyAsync(p, c->h.lev[l].theta, sizeof(float4) * c->h.lev[l].n3, cudaMemcpyDeviceToHost, s));
    p += sizeof(float4) * c->h.lev[l].n3;
    if (c->h.C == 6) {
      CU(c, cudaMemcpyAsync(p, c->h.lev[l].theta_t, sizeof(float4) * c->h.lev[l].n3, cudaMemcpyDeviceToHost, s));
      p += sizeof(float4) * c->h.lev[l].n3;
    }
  }
  CU(c, cudaStreamSynchronize(s));
  return PDG_OK;
}

pdg_status pdg_load_state(pdg_ctx* c, const void* host_buf, size_t n, void* cuda_stream) {
  if (!c || !host_buf) return PDG_ERR_INVALID;
  if (c->in_frame) return c->fail(PDG_ERR_STATE, "load only between frames");
  if (n < pdg_state_bytes(c)) return c->fail(PDG_ERR_INVALID, "state buffer too small");
  StateHeader hd;
  std::memcpy(&hd, host_buf, sizeof(hd));
  if (std::memcmp(hd.magic, "PDGSTAT", 8) != 0 || hd.version != 2 || hd.V != c->V || hd.L != c->h.L || hd.C != c->h.C ||
      hd.N < 1 || hd.N > c->max_pts)
    return c->fail(PDG_ERR_INVALID, "state does not match this context");
  for (int l = 0; l < c->h.L; ++l)
    if (hd.res[l] != c->h.lev[l].n) return c->fail(PDG_ERR_INVALID, "state does not match this context");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const char* p = (const char*)host_buf + sizeof(hd);
  CU(c, cudaMemcpyAsync(c->h.verts4, p, sizeof(float4) * c->V, cudaMemcpyHostToDevice, s));
  p += sizeof(float4) * c->V;
  CU(c, cudaMemcpyAsync(c->h.src4, p, sizeof(float4) * c->max_pts, cudaMemcpyHostToDevice, s));
  p += sizeof(float4) * c->max_pts;
  for (int l = 0; l < c->h.L; ++l) {
    CU(c, cudaMemcpyAsync(c->h.lev[l].theta, p, sizeof(float4) * c->h.lev[l].n3, cudaMemcpyHostToDevice, s));
    p += sizeof(float4) * c->h.lev[l].n3;
    if (c->h.C == 6) {
      CU(c, cudaMemcpyAsync(c->h.lev[l].theta_t, p, sizeof(float4) * c->h.lev[l].n3, cudaMemcpyHostToDevice, s));
      p += sizeof(float4) * c->h.lev[l].n3;
    }
  }
  c->h.N = hd.N;
  c->h.Q = c->V + hd.N;
  TRY(upload_job(c, s));
  CU(c, cudaStreamSynchronize(s));
  return PDG_OK;
}

}  // extern "C"
