// Batched solves: many independent diffusion problems of uneven size, each
// solved with FP32 V-cycles (Algorithm 1) inside FP64 iterative refinement,
// all advanced together.
//
// Organisation.  Every problem is set up as a hierarchy of its own.  The
// solve groups, for every grid side n, the levels of that side across all
// problems and runs each leg of the V-cycle (bmg_legs.cuh) as ONE launch over
// all of them, finest 5-point and coarse 9-point levels alike: the problem
// index is blockIdx.z, and a problem that has converged leaves at once.
// Levels of side 31 and below run in the shared-memory coarse kernel, one
// thread block per problem.  The FP64 work on the finest levels is one launch
// per pass over all problems, cut into units of some 4096 points, so that a
// 1023^2 problem gets the blocks its size asks for (64 blocks whatever the
// size took 18.7 us a pass, 47 % of a 48-problem solve).  Per-problem FP64
// residual norms and stop tests decide which problems stay active; the whole
// refinement loop is one CUDA graph whose WHILE node repeats while any
// problem is active.  V-cycles with other than one or two pre- and one
// post-smoothing sweep run one launch per operation and level class instead;
// their sweeps' tile shapes are chosen per level side by timing the
// candidates on the batch (autotuner, cached per process and optionally in
// the file named by BMG_TUNE_CACHE).
#include "bmg_krylov.cuh"
#include "bmg_legs.cuh"
#include "bmg_sweep_tile.cuh"

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace bmg {

namespace {

constexpr int kUnitRuns = 8;      // runs of kKT pairs a unit of FP64 work holds (4096 points)
constexpr int kNT = kKT;          // threads of the norm kernels
constexpr int kCoarseSide = 31;   // levels with side <= this: persistent kernel

inline int cdiv(long a, long b) { return int((a + b - 1) / b); }

// ---------------------------------------------------------------------------
// Batched V-cycle kernels (FP32).  z = blockIdx.z indexes the class members.
// ---------------------------------------------------------------------------

template <bool NINE, int TX, int TY, int NT>
__global__ void __launch_bounds__(NT) k_bsweep(const LevelV<float>* __restrict__ views,
                                               const int* __restrict__ pids,
                                               const Scalars* __restrict__ sc, unsigned order) {
  const int z = blockIdx.z;
  if (!sc[pids[z]].go) return;
  const LevelV<float> L = views[z];
  sweep_tile<float, NINE, TX, TY, NT>(L, L.x, L.x2, order, blockIdx.x, blockIdx.y);
}

template <bool NINE>
__global__ void k_bresid(const LevelV<float>* __restrict__ views, const int* __restrict__ pids,
                         const Scalars* __restrict__ sc) {
  const int z = blockIdx.z;
  if (!sc[pids[z]].go) return;
  const LevelV<float> L = views[z];
  const int i = blockIdx.x * blockDim.x + threadIdx.x + 1;
  const int j = blockIdx.y + 1;
  if (i > L.nx) return;
  const int o = j * L.pitch + i;
  L.r[o] = resid_value<float, NINE>(L, L.x, L.b[o], o);
}

__global__ void k_brestrict(const LevelV<float>* __restrict__ fine,
                            const LevelV<float>* __restrict__ coarse, const int* __restrict__ pids,
                            const Scalars* __restrict__ sc) {
  const int z = blockIdx.z;
  if (!sc[pids[z]].go) return;
  const LevelV<float> F = fine[z];
  const LevelV<float> Cc = coarse[z];
  const int I = blockIdx.x * blockDim.x + threadIdx.x + 1;
  const int J = blockIdx.y + 1;
  if (I > Cc.nx) return;
  const int c = J * Cc.pitch + I;
  Cc.b[c] = restrict_value<float>(F.P, Cc.pitch, F.r, F.pitch, c, 2 * J * F.pitch + 2 * I);
  Cc.x[c] = 0.0f;
}

__global__ void k_binterp(const LevelV<float>* __restrict__ fine,
                          const LevelV<float>* __restrict__ coarse, const int* __restrict__ pids,
                          const Scalars* __restrict__ sc, int out_of_place) {
  const int z = blockIdx.z;
  if (!sc[pids[z]].go) return;
  const LevelV<float> F = fine[z];
  const float* xc = coarse[z].x;
  const int i = blockIdx.x * blockDim.x + threadIdx.x + 1;
  const int j = blockIdx.y + 1;
  if (i > F.nx) return;
  const int o = j * F.pitch + i;
  const float v = F.x[o] + interp_value<float>(F.P, F.cpitch, xc, i, j);
  (out_of_place ? F.x2 : F.x)[o] = v;
}

// The legs of the levels of one side: the z-th member's iterate goes
// x -> x2 -> x.  Its iterate is zero on entry (every level's is: the finest
// level solves for a correction).  Whether a problem is active was settled
// before the kernel that precedes this one began, so it is read, and the
// operator staged, ahead of the wait; a block that leaves waits all the same,
// because the kernel that follows relies on this one to have waited.
template <bool NINE, int NS, int TX, int TY, int NT>
__device__ __forceinline__ void batch_down(const LevelV<float>& F, const LevelV<float>& Cc, float* sm) {
  float pw[8];
  down_constants<float, NINE, NS, TX, TY, NT>(F, Cc, sm, blockIdx.x, blockIdx.y, pw);
  griddep_wait();
  down_tile<float, NINE, NS, true, TX, TY, NT>(F, F.x, F.x2, Cc, sm, blockIdx.x, blockIdx.y, pw);
}
template <int NS, int TX, int TY, int NT>
__global__ void __launch_bounds__(NT) k_bdown(const LevelV<float>* __restrict__ fine,
                                              const LevelV<float>* __restrict__ coarse,
                                              const int* __restrict__ pids,
                                              const Scalars* __restrict__ sc) {
  extern __shared__ __align__(16) unsigned char leg_smem[];
  float* sm = reinterpret_cast<float*>(leg_smem);
  const int z = blockIdx.z;
  if (!sc[pids[z]].go) {
    griddep_wait();
    return;
  }
  const LevelV<float> F = fine[z], Cc = coarse[z];
  if (F.SW)
    batch_down<true, NS, TX, TY, NT>(F, Cc, sm);
  else
    batch_down<false, NS, TX, TY, NT>(F, Cc, sm);
}

template <bool NINE, int TX, int TY, int NT>
__device__ __forceinline__ void batch_up(const LevelV<float>& F, const float* xc, float* sm) {
  float w[8];
  up_constants<float, NINE, TX, TY, NT, false>(F, sm, blockIdx.x, blockIdx.y, w);
  griddep_wait();
  up_tile<float, NINE, TX, TY, NT, false>(F, F.x2, xc, F.x, nullptr, sm, blockIdx.x, blockIdx.y, w);
}
template <int TX, int TY, int NT>
__global__ void __launch_bounds__(NT) k_bup(const LevelV<float>* __restrict__ fine,
                                            const LevelV<float>* __restrict__ coarse,
                                            const int* __restrict__ pids, const Scalars* __restrict__ sc) {
  extern __shared__ __align__(16) unsigned char leg_smem[];
  float* sm = reinterpret_cast<float*>(leg_smem);
  const int z = blockIdx.z;
  if (!sc[pids[z]].go) {
    griddep_wait();
    return;
  }
  const LevelV<float> F = fine[z];
  if (F.SW)
    batch_up<true, TX, TY, NT>(F, coarse[z].x, sm);
  else
    batch_up<false, TX, TY, NT>(F, coarse[z].x, sm);
}

// ---------------------------------------------------------------------------
// FP64 work on the problems' finest levels: a block per unit.
// ---------------------------------------------------------------------------

struct BUnit {
  int p, local, count;           // problem, unit of it, its units
};
struct BSpan {
  int first, count;              // a problem's units
};
// Per problem: its finest levels and CG vectors.
struct BProb {
  LevelV<double> d;
  LevelV<float> f;
  PcgVec v;
};

// what == 0: partial sums of b^2.  what == 1 (active problems only): r = b -
// A x in FP64, partial sums of r^2, FP32 right-hand side r / ||r_prev||
// (zero_x: and a zero FP32 iterate, for cycles that read it).
template <int WHAT>
__global__ void __launch_bounds__(kKT) k_brefine_resid(const BProb* __restrict__ prob,
                                                       const BUnit* __restrict__ units,
                                                       const Scalars* __restrict__ sc, int zero_x,
                                                       double* __restrict__ partials) {
  griddep_wait();
  const BUnit u = units[blockIdx.x];
  if (WHAT == 1 && !sc[u.p].go) return;
  const LevelV<double>& L = prob[u.p].d;
  const LevelV<float>& F = prob[u.p].f;
  const double inv = WHAT ? sc[u.p].inv : 0.0;
  // FP32 scaling of the right-hand side, as in the single-problem kernel
  const bool fp32_scale = inv > 1e-28 && inv < 1e28;
  const float inv32 = float(inv);
  double acc = 0.0;
  for_pairs(L.nx, L.ny, u.local, u.count, [&](int j, int i, bool two) {
    const int o = j * L.pitch + i;
    const double2 bv = load2(L.b + o);
    if (WHAT == 0) {
      acc = fma(bv.x, bv.x, acc);
      if (two) acc = fma(bv.y, bv.y, acc);
      return;
    }
    const double2 r = resid_pair(load_resid(L, L.x, o), bv);
    acc = fma(r.x, r.x, acc);
    const int of = j * F.pitch + i;
    const float f0 = fp32_scale ? to_float(r.x) * inv32 : to_float(r.x * inv);
    F.b[of] = f0;
    if (zero_x) F.x[of] = 0.0f;
    if (two) {
      acc = fma(r.y, r.y, acc);
      F.b[of + 1] = fp32_scale ? to_float(r.y) * inv32 : to_float(r.y * inv);
      if (zero_x) F.x[of + 1] = 0.0f;
    }
  });
  acc = krylov_block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// One block per problem: sums its partials and applies the stop test; the
// last block to finish knows whether any problem is still active, and drives
// the graph's WHILE node (`count`: problems done and active, back to zero).
__global__ void __launch_bounds__(kNT) k_bnorm_final(const double* __restrict__ partials,
                                                     const BSpan* __restrict__ spans,
                                                     Scalars* __restrict__ sc, int what,
                                                     cudaGraphConditionalHandle handle, int use_handle,
                                                     int* __restrict__ count) {
  griddep_wait();
  const int p = blockIdx.x;
  Scalars* s = sc + p;
  int go = 0;
  if (what == 0 || s->go) {
    double acc = 0.0;
    const BSpan q = spans[p];
    for (int k = threadIdx.x; k < q.count; k += kNT) acc += partials[q.first + k];
    acc = krylov_block_sum(acc);
    if (threadIdx.x == 0) {
      if (what == 0) {
        s->bnorm2 = acc;
        s->rnorm2 = acc;
        s->rnorm = sqrt(acc);
        s->inv = acc > 0.0 ? 1.0 / s->rnorm : 0.0;
        go = acc > 0.0 ? 1 : 0;     // a zero right-hand side needs no cycle
        s->go = go;
        s->rel = 0.0;
      } else {
        s->scale2 = s->rnorm2;
        s->scale = sqrt(s->scale2);
        s->rnorm2 = acc;
        s->rnorm = sqrt(acc);
        s->inv = acc > 0.0 ? 1.0 / s->rnorm : 0.0;
        const double rel = sqrt(acc / s->bnorm2);
        s->rel = rel;
        const bool finite = isfinite(rel);
        if (!finite) s->err |= DEV_NAN;
        go = (finite && rel > s->tol && s->cycles < s->max_cycles && s->err == 0) ? 1 : 0;
        s->go = go;
        s->cycles += go;
      }
    }
  }
  if (threadIdx.x != 0) return;
  if (go) atomicAdd(&count[1], 1);
  __threadfence();
  if (atomicAdd(&count[0], 1) == int(gridDim.x) - 1) {
    const int any = atomicExch(&count[1], 0);
    count[0] = 0;
    if (use_handle) cudaGraphSetConditional(handle, any ? 1u : 0u);
  }
}

__global__ void __launch_bounds__(kKT) k_bupdate(const BProb* __restrict__ prob,
                                                 const BUnit* __restrict__ units,
                                                 const Scalars* __restrict__ sc) {
  griddep_wait();
  const BUnit u = units[blockIdx.x];
  if (!sc[u.p].go) return;
  const LevelV<double>& L = prob[u.p].d;
  const LevelV<float>& F = prob[u.p].f;
  const double s = sc[u.p].scale;
  for_pairs(L.nx, L.ny, u.local, u.count, [&](int j, int i, bool two) {
    const int o = j * L.pitch + i;
    const double2 x = load2(L.x + o);
    const float2 e = *reinterpret_cast<const float2*>(F.x + j * F.pitch + i);
    store2(L.x + o, fma(s, to_double(e.x), x.x), fma(s, to_double(e.y), x.y), two);
  });
}

// ---------------------------------------------------------------------------
// Batched conjugate gradients (BMG_SOLVER_PCG): per problem, CG on its finest
// operator in FP64, preconditioned by one symmetric FP32 V(nu, nu) cycle of
// the batched V-cycle (r / ||r|| cast to the FP32 finest level, z = ||r|| e),
// in the single-problem solver's order and with its passes (bmg_krylov.cuh).
// Active problems only.
// ---------------------------------------------------------------------------

template <int WHAT>
__global__ void __launch_bounds__(kKT) k_bpcg(const BProb* __restrict__ prob,
                                              const BUnit* __restrict__ units,
                                              const Scalars* __restrict__ sc,
                                              double* __restrict__ partials) {
  griddep_wait();
  const BUnit u = units[blockIdx.x];
  if (!sc[u.p].go) return;
  const BProb& q = prob[u.p];
  double s = krylov_pass<WHAT, true>(q.d, &q.f, q.v, sc + u.p, false, u.local, u.count);
  if (WHAT == K_P) return;
  s = krylov_block_sum(s);
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

__global__ void __launch_bounds__(kKT) k_bpcg_cast(const BProb* __restrict__ prob,
                                                   const BUnit* __restrict__ units,
                                                   const Scalars* __restrict__ sc, int zero_x) {
  griddep_wait();
  const BUnit u = units[blockIdx.x];
  if (!sc[u.p].go) return;
  krylov_cast(prob[u.p].d, prob[u.p].f, sc + u.p, zero_x != 0, u.local, u.count);
}

// One block per problem: AP alpha = rz / sum (0 for a zero denominator); RZ
// beta = sum / rz (0 while rz is 0: the first direction is z), rz = sum.
__global__ void __launch_bounds__(kNT) k_bpcg_scalar(const double* __restrict__ partials,
                                                     const BSpan* __restrict__ spans,
                                                     Scalars* __restrict__ sc, int what) {
  griddep_wait();
  const int pr = blockIdx.x;
  Scalars* s = sc + pr;
  if (!s->go) return;
  double acc = 0.0;
  const BSpan q = spans[pr];
  for (int k = threadIdx.x; k < q.count; k += kNT) acc += partials[q.first + k];
  acc = krylov_block_sum(acc);
  if (threadIdx.x != 0) return;
  if (what == K_AP) {
    s->alpha = acc != 0.0 ? s->rz / acc : 0.0;
  } else {
    acc *= s->rnorm;   // (the partials are of r.e, z = ||r|| e)
    s->beta = s->rz != 0.0 ? acc / s->rz : 0.0;
    s->rz = acc;
  }
}

// Dense user arrays <-> the finest planes, all problems in one launch (their
// b, then their x, in `user`).  In: the right-hand side into the level's b
// plane and the iterate into its x plane, or (pcg) into the CG vectors, b into
// both.  Out: the iterate; a problem with a zero right-hand side runs no cycle
// and has the solution 0.
__global__ void __launch_bounds__(kKT) k_bpack(const BProb* __restrict__ prob,
                                               const BUnit* __restrict__ units,
                                               double* const* __restrict__ user, int nprob, int pcg) {
  const BUnit u = units[blockIdx.x];
  const BProb& q = prob[u.p];
  const LevelV<double>& L = q.d;
  const double* __restrict__ b = user[u.p];
  const double* __restrict__ x = user[nprob + u.p];
  for_pairs(L.nx, L.ny, u.local, u.count, [&](int j, int i, bool two) {
    const size_t e = size_t(j - 1) * L.nx + i - 1;
    const int o = j * L.pitch + i;
    const double b0 = b[e], x0 = x[e], b1 = two ? b[e + 1] : 0.0, x1 = two ? x[e + 1] : 0.0;
    store2(L.b + o, b0, b1, two);
    if (pcg) store2(q.v.b + o, b0, b1, two);
    store2((pcg ? q.v.x : L.x) + o, x0, x1, two);
  });
}

__global__ void __launch_bounds__(kKT) k_bunpack(const BProb* __restrict__ prob,
                                                 const BUnit* __restrict__ units,
                                                 const Scalars* __restrict__ sc,
                                                 double* const* __restrict__ user, int nprob, int pcg) {
  const BUnit u = units[blockIdx.x];
  const BProb& q = prob[u.p];
  const LevelV<double>& L = q.d;
  double* __restrict__ x = user[nprob + u.p];
  const bool zero = sc[u.p].bnorm2 == 0.0;
  for_pairs(L.nx, L.ny, u.local, u.count, [&](int j, int i, bool two) {
    const size_t e = size_t(j - 1) * L.nx + i - 1;
    const double2 v = load2((pcg ? q.v.x : L.x) + j * L.pitch + i);
    x[e] = zero ? 0.0 : v.x;
    if (two) x[e + 1] = zero ? 0.0 : v.y;
  });
}

// ---------------------------------------------------------------------------
// Tile variants of the batched sweep and their autotuner.
// ---------------------------------------------------------------------------

constexpr int kTileVariants = 3;   // 32x16/128 threads, 64x16/256, 128x32/256

void launch_bsweep(int variant, bool nine, int n, int count, const LevelV<float>* views,
                   const int* pids, const Scalars* sc, unsigned order, cudaStream_t s) {
#define BMG_BSWEEP(TX, TY, NT)                                                          \
  do {                                                                                  \
    const dim3 grid(cdiv(n, TX), cdiv(n, TY), count);                                   \
    if (nine)                                                                           \
      launch_plain(k_bsweep<true, TX, TY, NT>, grid, dim3(NT), 0, s, views, pids, sc, order);  \
    else                                                                                \
      launch_plain(k_bsweep<false, TX, TY, NT>, grid, dim3(NT), 0, s, views, pids, sc, order); \
  } while (0)
  switch (variant) {
    case 0: BMG_BSWEEP(32, 16, 128); break;
    case 1: BMG_BSWEEP(64, 16, 256); break;
    default: BMG_BSWEEP(128, 32, 256); break;
  }
#undef BMG_BSWEEP
  count_launch();
}

std::mutex g_tune_mu;
std::map<std::string, int> g_tune;   // "device/n/kind/count" -> variant
bool g_tune_loaded = false;

std::string tune_key(int n, bool nine, int count) {
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceProp prop;
  cudaGetDeviceProperties(&prop, dev);
  char buf[256];
  std::snprintf(buf, sizeof(buf), "%s/%d/%d/%d", prop.name, n, nine ? 9 : 5, count);
  std::string k(buf);
  for (char& c : k)
    if (c == ' ') c = '_';
  return k;
}

void tune_load() {
  if (g_tune_loaded) return;
  g_tune_loaded = true;
  const char* path = std::getenv("BMG_TUNE_CACHE");
  if (!path) return;
  FILE* f = std::fopen(path, "r");
  if (!f) return;
  char key[256];
  int v;
  while (std::fscanf(f, "%255s %d", key, &v) == 2) g_tune[key] = v;
  std::fclose(f);
}

void tune_store(const std::string& key, int v) {
  g_tune[key] = v;
  const char* path = std::getenv("BMG_TUNE_CACHE");
  if (!path) return;
  FILE* f = std::fopen(path, "a");
  if (!f) return;
  std::fprintf(f, "%s %d\n", key.c_str(), v);
  std::fclose(f);
}

}  // namespace

// ---------------------------------------------------------------------------
// Batch object
// ---------------------------------------------------------------------------

struct BClass {                  // levels of one side and one kind across problems
  int n = 0;
  bool nine = false;
  int count = 0;
  int tile = 1;
  int* pids = nullptr;                       // device
  LevelV<float>* view[2] = {nullptr, nullptr};   // parity 0: (x, x2); 1: swapped
  LevelV<float>* coarse = nullptr;           // next coarser level of the same problems
  int parity_after_pre = 0;
};

struct Batch {
  int nprob = 0;
  bmg_options opt{};
  std::vector<Hierarchy*> hs;
  std::vector<int> side;
  std::vector<BClass> cls;       // descending side; per side 5-point first
  std::vector<BClass> sides;     // descending side, both kinds together
  Scalars* sc = nullptr;
  Scalars* sc_host = nullptr;
  double* partials = nullptr;
  BProb* prob = nullptr;
  double** user = nullptr;       // the callers' b, then x
  BUnit* units = nullptr;
  BSpan* spans = nullptr;
  int nunits = 0;
  unsigned char* coarse_args = nullptr;   // of the shared-memory coarse kernel
  size_t coarse_bytes = 0;
  int* count = nullptr;          // problems done and active (k_bnorm_final)
  bool legs = false;             // fused legs (one or two pre-, one post-sweep)
  void* arena = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaGraphConditionalHandle handle = 0;
  double setup_ms = 0.0;
};

namespace {

template <typename T>
T* carve(char*& p, size_t n) {
  T* r = reinterpret_cast<T*>(p);
  p += ((n * sizeof(T) + 255) / 256) * 256;
  return r;
}

// failed: work of a call that failed may be under way on the hierarchies.
void destroy_batch(Batch* b, bool failed = false) {
  if (!b) return;
  if (failed)
    for (Hierarchy* h : b->hs) h->pending.lost();
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  for (Hierarchy* h : b->hs) free_hierarchy(h);
  if (b->arena) cudaFree(b->arena);
  if (b->sc_host) cudaFreeHost(b->sc_host);
  delete b;
}

// Tiles of a side's legs: the largest that still give every SM two blocks.
template <int TX, int TY>
int side_tiles(const BClass& c) { return cdiv(c.n, TX) * cdiv(c.n, TY) * c.count; }

// A kernel serves finest and coarse levels; its shared memory is the larger.
template <int NS, int TX, int TY>
constexpr size_t bdown_smem() {
  return std::max(DownLeg<float, true, NS, TX, TY>::SMEM, DownLeg<float, false, NS, TX, TY>::SMEM);
}
template <int TX, int TY>
constexpr size_t bup_smem() {
  return std::max(UpLeg<float, true, TX, TY, false>::SMEM, UpLeg<float, false, TX, TY, false>::SMEM);
}
template <int TX, int TY, int NT>
bool bleg_ready() {
  return use_shared(k_bdown<1, TX, TY, NT>, bdown_smem<1, TX, TY>()) &&
         use_shared(k_bdown<2, TX, TY, NT>, bdown_smem<2, TX, TY>()) &&
         use_shared(k_bup<TX, TY, NT>, bup_smem<TX, TY>());
}
bool blegs_ready() { return bleg_ready<32, 16, 256>() && bleg_ready<16, 8, 128>() && bleg_ready<8, 8, 128>(); }

template <int NS, int TX, int TY, int NT>
void launch_bdown(const BClass& c, const Scalars* sc, cudaStream_t s) {
  constexpr size_t smem = bdown_smem<NS, TX, TY>();
  launch_pdl(k_bdown<NS, TX, TY, NT>, dim3(cdiv(c.n, TX), cdiv(c.n, TY), c.count), dim3(NT), smem, s,
             (const LevelV<float>*)c.view[0], (const LevelV<float>*)c.coarse, (const int*)c.pids, sc);
  count_launch();
}
template <int TX, int TY, int NT>
void launch_bup(const BClass& c, const Scalars* sc, cudaStream_t s) {
  constexpr size_t smem = bup_smem<TX, TY>();
  launch_pdl(k_bup<TX, TY, NT>, dim3(cdiv(c.n, TX), cdiv(c.n, TY), c.count), dim3(NT), smem, s,
             (const LevelV<float>*)c.view[0], (const LevelV<float>*)c.coarse, (const int*)c.pids, sc);
  count_launch();
}
template <int TX, int TY, int NT>
void launch_bleg(const BClass& c, int ns, const Scalars* sc, cudaStream_t s) {
  if (ns == 0)
    launch_bup<TX, TY, NT>(c, sc, s);
  else if (ns == 1)
    launch_bdown<1, TX, TY, NT>(c, sc, s);
  else
    launch_bdown<2, TX, TY, NT>(c, sc, s);
}
// ns pre-sweeps of the down leg, 0: the up leg.
void launch_side(const BClass& c, int ns, const Scalars* sc, cudaStream_t s) {
  if (side_tiles<32, 16>(c) >= 2 * 152)
    launch_bleg<32, 16, 256>(c, ns, sc, s);
  else if (side_tiles<16, 8>(c) >= 2 * 152)
    launch_bleg<16, 8, 128>(c, ns, sc, s);
  else
    launch_bleg<8, 8, 128>(c, ns, sc, s);
}

void launch_bcoarse(Batch* b, cudaStream_t s) {
  launch_coarse_smem_batch(b->coarse_args, b->nprob, b->coarse_bytes, b->sc, s);
}

// Downward half of the batched V-cycle, coarse kernel, upward half.
void enqueue_bvcycle(Batch* b, cudaStream_t s) {
  const int nu1 = b->opt.nu1, nu2 = b->opt.nu2;
  if (b->legs) {
    for (const BClass& c : b->sides) launch_side(c, nu1, b->sc, s);
    launch_bcoarse(b, s);
    for (auto it = b->sides.rbegin(); it != b->sides.rend(); ++it) launch_side(*it, 0, b->sc, s);
    return;
  }
  const bool oop = ((nu1 + nu2) & 1) != 0;
  for (BClass& c : b->cls) {
    int par = 0;
    for (int k = 0; k < nu1; ++k) {
      launch_bsweep(c.tile, c.nine, c.n, c.count, c.view[par], c.pids, b->sc,
                    c.nine ? four_order(false) : rb_order(false), s);
      par ^= 1;
    }
    const dim3 g(cdiv(c.n, 128), c.n, c.count);
    if (c.nine)
      launch_plain(k_bresid<true>, g, dim3(128), 0, s, c.view[par], c.pids, b->sc);
    else
      launch_plain(k_bresid<false>, g, dim3(128), 0, s, c.view[par], c.pids, b->sc);
    const int nc = (c.n - 1) / 2;
    launch_plain(k_brestrict, dim3(cdiv(nc, 128), nc, c.count), dim3(128), 0, s, c.view[par], c.coarse, c.pids,
                 b->sc);
    count_launch(2);
    c.parity_after_pre = par;
  }
  launch_bcoarse(b, s);
  for (auto it = b->cls.rbegin(); it != b->cls.rend(); ++it) {
    BClass& c = *it;
    int par = c.parity_after_pre;
    launch_plain(k_binterp, dim3(cdiv(c.n, 128), c.n, c.count), dim3(128), 0, s, c.view[par], c.coarse, c.pids,
                 b->sc, oop ? 1 : 0);
    count_launch();
    if (oop) par ^= 1;
    for (int k = 0; k < nu2; ++k) {
      launch_bsweep(c.tile, c.nine, c.n, c.count, c.view[par], c.pids, b->sc,
                    c.nine ? four_order(true) : rb_order(true), s);
      par ^= 1;
    }
  }
}

void launch_bnorm_final(Batch* b, int what, bool use_handle, cudaStream_t s) {
  launch_pdl(k_bnorm_final, dim3(b->nprob), dim3(kNT), 0, s, (const double*)b->partials,
             (const BSpan*)b->spans, b->sc, what, b->handle, use_handle ? 1 : 0, b->count);
  count_launch();
}

void enqueue_residuals(Batch* b, int what, bool use_handle, cudaStream_t s) {
  if (what == 0)
    launch_pdl(k_brefine_resid<0>, dim3(b->nunits), dim3(kKT), 0, s, (const BProb*)b->prob,
               (const BUnit*)b->units, (const Scalars*)b->sc, 0, b->partials);
  else
    launch_pdl(k_brefine_resid<1>, dim3(b->nunits), dim3(kKT), 0, s, (const BProb*)b->prob,
               (const BUnit*)b->units, (const Scalars*)b->sc, b->legs ? 0 : 1, b->partials);
  count_launch();
  launch_bnorm_final(b, what, use_handle, s);
}

void enqueue_update(Batch* b, cudaStream_t s) {
  launch_pdl(k_bupdate, dim3(b->nunits), dim3(kKT), 0, s, (const BProb*)b->prob, (const BUnit*)b->units,
             (const Scalars*)b->sc);
  count_launch();
}

template <int WHAT>
void enqueue_pcg_vec(Batch* b, cudaStream_t s) {
  launch_pdl(k_bpcg<WHAT>, dim3(b->nunits), dim3(kKT), 0, s, (const BProb*)b->prob, (const BUnit*)b->units,
             (const Scalars*)b->sc, b->partials);
  count_launch();
}

void enqueue_pcg_scalar(Batch* b, int what, cudaStream_t s) {
  launch_pdl(k_bpcg_scalar, dim3(b->nprob), dim3(kNT), 0, s, (const double*)b->partials,
             (const BSpan*)b->spans, b->sc, what);
  count_launch();
}

// The first residual of PCG (r = B - A X) and its stop test.
void enqueue_pcg_init(Batch* b, cudaStream_t s) {
  enqueue_pcg_vec<K_INIT>(b, s);
  launch_bnorm_final(b, 1, false, s);
}

// One batched PCG iteration of the active problems: z = M^{-1} r (the FP32
// batched V-cycle after the cast), r.z and beta, p = z + beta p, q = A p and
// alpha, x += alpha p and r -= alpha q, the stop test.
void enqueue_pcg_iter(Batch* b, bool use_handle, cudaStream_t s) {
  launch_pdl(k_bpcg_cast, dim3(b->nunits), dim3(kKT), 0, s, (const BProb*)b->prob, (const BUnit*)b->units,
             (const Scalars*)b->sc, b->legs ? 0 : 1);
  count_launch();
  enqueue_bvcycle(b, s);
  enqueue_pcg_vec<K_RZ>(b, s);
  enqueue_pcg_scalar(b, K_RZ, s);
  enqueue_pcg_vec<K_P>(b, s);
  enqueue_pcg_vec<K_AP>(b, s);
  enqueue_pcg_scalar(b, K_AP, s);
  enqueue_pcg_vec<K_XR>(b, s);
  launch_bnorm_final(b, 1, use_handle, s);
}

// Pick the fastest tile variant of every class by timing sweeps on the batch
// (x = 0 and b = 0 after setup, so the timing sweeps change nothing).
int autotune(Batch* b, cudaStream_t s) {
  std::lock_guard<std::mutex> g(g_tune_mu);
  tune_load();
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return BMG_ECUDA;
  // every problem must count as active while timing
  for (int p = 0; p < b->nprob; ++p) b->sc_host[p] = Scalars{};
  std::vector<Scalars> act(b->nprob);
  for (auto& a : act) a.go = 1;
  cudaMemcpyAsync(b->sc, act.data(), sizeof(Scalars) * b->nprob, cudaMemcpyHostToDevice, s);
  for (BClass& c : b->cls) {
    const std::string key = tune_key(c.n, c.nine, c.count);
    auto it = g_tune.find(key);
    if (it != g_tune.end()) {
      c.tile = it->second;
      continue;
    }
    float best = 1e30f;
    int bv = 1;
    for (int v = 0; v < kTileVariants; ++v) {
      const unsigned order = c.nine ? four_order(false) : rb_order(false);
      launch_bsweep(v, c.nine, c.n, c.count, c.view[0], c.pids, b->sc, order, s);
      cudaEventRecord(e0, s);
      for (int r = 0; r < 3; ++r)
        launch_bsweep(v, c.nine, c.n, c.count, c.view[0], c.pids, b->sc, order, s);
      cudaEventRecord(e1, s);
      cudaEventSynchronize(e1);
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (ms < best) {
        best = ms;
        bv = v;
      }
    }
    c.tile = bv;
    tune_store(key, bv);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return cudaGetLastError() == cudaSuccess ? BMG_OK : BMG_ECUDA;
}

// The refinement loop as one graph: WHILE(any active) { V-cycle; update;
// residuals + stop tests + any }, or (BMG_SOLVER_PCG) WHILE(any active) {
// one PCG iteration }.  Recording executes nothing.
int build_graph(Batch* b) {
  if (cudaGraphCreate(&b->graph, 0) != cudaSuccess) return BMG_ECUDA;
  if (cudaGraphConditionalHandleCreate(&b->handle, b->graph, 1, cudaGraphCondAssignDefault) !=
      cudaSuccess)
    return BMG_ECUDA;
  cudaGraph_t body = nullptr;
  {
    GraphRecorder rec(b->graph);
    body = rec.loop(b->handle);
  }
  if (!body) return BMG_ECUDA;
  {
    GraphRecorder rec(body);
    if (b->opt.solver == BMG_SOLVER_PCG) {
      enqueue_pcg_iter(b, true, nullptr);
    } else {
      enqueue_bvcycle(b, nullptr);
      enqueue_update(b, nullptr);
      enqueue_residuals(b, 1, true, nullptr);
    }
    if (!rec.ok()) return BMG_ECUDA;
  }
  return cudaGraphInstantiate(&b->exec, b->graph, 0) == cudaSuccess ? BMG_OK : BMG_ECUDA;
}

double now_ms() {
  return std::chrono::duration<double, std::milli>(
             std::chrono::steady_clock::now().time_since_epoch())
      .count();
}

}  // namespace

}  // namespace bmg

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------

using bmg::Batch;

extern "C" int bmg_batch_setup(int nprob, const double* const* k_dev, const int* n,
                               const bmg_options* opt_in, bmg_stream_t stream, bmg_batch** out) {
  using namespace bmg;
  if (!out) return BMG_EINVAL;
  *out = nullptr;
  if (nprob < 1 || !k_dev || !n) return BMG_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const double t0 = now_ms();
  bmg_options opt;
  bmg_default_options(&opt);
  if (opt_in) opt = *opt_in;
  if (opt.smoother != BMG_SMOOTH_POINT) {
    set_last_error("batch setup: only the point smoother is batched");
    return BMG_EINVAL;
  }
  if (opt.solver == BMG_SOLVER_PCG && (opt.nu1 != opt.nu2 || opt.interp_residual_term)) {
    set_last_error("batch setup: BMG_SOLVER_PCG needs nu1 == nu2 and interp_residual_term == 0");
    return BMG_EINVAL;
  }
  if (opt.solver != BMG_SOLVER_VCYCLE && opt.solver != BMG_SOLVER_PCG) return BMG_EINVAL;
  opt.precision = BMG_FP32_REFINE;
  Batch* b = new Batch();
  b->nprob = nprob;
  b->opt = opt;
  auto fail = [&](int code) {
    destroy_batch(b, code == BMG_ECUDA);
    return code;
  };
  // individual hierarchies (threshold: levels of side <= 31 in the coarse kernel)
  for (int p = 0; p < nprob; ++p) {
    // batched problems: square, sides 2^m - 1 (the level classes below rely on it)
    if (!k_dev[p] || n[p] < 3 || ((n[p] + 1) & n[p]) != 0) return fail(BMG_EINVAL);
    int levels_small = 0;
    for (int m = n[p]; m >= 3; m = (m - 1) / 2)
      if (m <= kCoarseSide) ++levels_small;
    bmg_options o = opt;
    o.coarse_threshold = std::max(1, levels_small);
    o.coarse_ctas = 1;         // the batched coarse kernel runs one block per problem
    Hierarchy* h = nullptr;
    const int rc = setup_impl(k_dev[p], n[p], n[p], &o, s, &h);
    if (rc) {
      set_last_error("batch setup: problem %d: %s", p, bmg_last_error());
      return fail(rc);
    }
    b->hs.push_back(h);
    b->side.push_back(n[p]);
  }
  // classes: for each side > kCoarseSide, the 5-point finest levels and the
  // 9-point levels of larger problems
  std::vector<int> sides;
  for (int v : b->side)
    for (int m = v; m > kCoarseSide; m = (m - 1) / 2) sides.push_back(m);
  std::sort(sides.begin(), sides.end(), std::greater<int>());
  sides.erase(std::unique(sides.begin(), sides.end()), sides.end());
  struct HostClass {
    BClass c;
    std::vector<int> pids;
    std::vector<LevelV<float>> v0, v1, vc;
  };
  if (!coarse_smem_batch_ready()) return fail(BMG_ECUDA);
  b->legs = (opt.nu1 == 1 || opt.nu1 == 2) && opt.nu2 == 1 && blegs_ready();
  std::vector<HostClass> hc;
  for (int m : sides) {
    // legs: one class per side (kind 2); else one per side and kind
    for (int kind = b->legs ? 2 : 0; kind < (b->legs ? 3 : 2); ++kind) {
      HostClass x;
      x.c.n = m;
      x.c.nine = kind == 1;
      for (int p = 0; p < nprob; ++p) {
        const Hierarchy* h = b->hs[p];
        const bool finest = b->side[p] == m;
        if (b->side[p] < m || (kind < 2 && finest == x.c.nine)) continue;
        int l = h->L - 1;
        while (h->f[l].nx != m) --l;
        LevelV<float> a = h->f[l], bb = h->f[l];
        std::swap(bb.x, bb.x2);
        x.pids.push_back(p);
        x.v0.push_back(a);
        x.v1.push_back(bb);
        x.vc.push_back(h->f[l - 1]);
      }
      x.c.count = int(x.pids.size());
      if (x.c.count) hc.push_back(std::move(x));
    }
  }
  // device arena for the descriptors
  size_t bytes = 0;
  auto al = [](size_t v) { return ((v + 255) / 256) * 256; };
  for (auto& x : hc) bytes += al(sizeof(int) * x.c.count) + 3 * al(sizeof(LevelV<float>) * x.c.count);
  // units of FP64 work, by problem
  std::vector<BUnit> units;
  std::vector<BSpan> spans;
  for (int p = 0; p < nprob; ++p) {
    const int k = cdiv(pair_runs(n[p], n[p]), kUnitRuns);
    spans.push_back(BSpan{int(units.size()), k});
    for (int i = 0; i < k; ++i) units.push_back(BUnit{p, i, k});
  }
  b->nunits = int(units.size());
  std::vector<unsigned char> cargs;
  coarse_smem_batch_args(b->hs[0], nullptr, cargs);
  const size_t cargs_one = cargs.size();
  bytes += al(sizeof(Scalars) * nprob) + al(sizeof(double) * b->nunits) + al(sizeof(BProb) * nprob) +
           al(sizeof(BUnit) * b->nunits) + al(sizeof(BSpan) * nprob) + al(cargs_one * nprob) +
           al(2 * sizeof(int)) + al(2 * sizeof(double*) * nprob);
  if (device_malloc(&b->arena, bytes) != cudaSuccess) return fail(BMG_ENOMEM);
  if (cudaMallocHost(&b->sc_host, sizeof(Scalars) * nprob) != cudaSuccess) return fail(BMG_ENOMEM);
  char* cur = static_cast<char*>(b->arena);
  for (auto& x : hc) {
    BClass c = x.c;
    c.pids = carve<int>(cur, c.count);
    c.view[0] = carve<LevelV<float>>(cur, c.count);
    c.view[1] = carve<LevelV<float>>(cur, c.count);
    c.coarse = carve<LevelV<float>>(cur, c.count);
    cudaMemcpyAsync(c.pids, x.pids.data(), sizeof(int) * c.count, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(c.view[0], x.v0.data(), sizeof(LevelV<float>) * c.count, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(c.view[1], x.v1.data(), sizeof(LevelV<float>) * c.count, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(c.coarse, x.vc.data(), sizeof(LevelV<float>) * c.count, cudaMemcpyHostToDevice, s);
    (b->legs ? b->sides : b->cls).push_back(c);
  }
  b->sc = carve<Scalars>(cur, nprob);
  b->partials = carve<double>(cur, b->nunits);
  b->prob = carve<BProb>(cur, nprob);
  b->units = carve<BUnit>(cur, b->nunits);
  b->spans = carve<BSpan>(cur, nprob);
  b->coarse_args = carve<unsigned char>(cur, cargs_one * nprob);
  b->count = carve<int>(cur, 2);
  b->user = carve<double*>(cur, 2 * nprob);
  std::vector<BProb> probs;
  cargs.clear();
  for (int p = 0; p < nprob; ++p) {
    const Hierarchy* h = b->hs[p];
    probs.push_back(BProb{h->d.back(), h->f.back(), PcgVec{h->pcg_x, h->pcg_b, h->pcg_p, h->pcg_q}});
    b->coarse_bytes = std::max(b->coarse_bytes, coarse_smem_batch_args(h, &b->sc[p].err, cargs));
    if (!h->coarse_smem) return fail(BMG_ECUDA);   // (levels of side <= 31 always fit)
  }
  cudaMemcpyAsync(b->prob, probs.data(), sizeof(BProb) * nprob, cudaMemcpyHostToDevice, s);
  cudaMemcpyAsync(b->units, units.data(), sizeof(BUnit) * units.size(), cudaMemcpyHostToDevice, s);
  cudaMemcpyAsync(b->spans, spans.data(), sizeof(BSpan) * nprob, cudaMemcpyHostToDevice, s);
  cudaMemcpyAsync(b->coarse_args, cargs.data(), cargs.size(), cudaMemcpyHostToDevice, s);
  cudaMemsetAsync(b->count, 0, 2 * sizeof(int), s);
  if (cudaStreamSynchronize(s) != cudaSuccess) return fail(BMG_ECUDA);
  int rc = b->legs ? BMG_OK : autotune(b, s);
  if (rc) return fail(rc);
  if ((rc = build_graph(b))) {
    set_last_error("batch setup: building the CUDA graph failed (%s)",
                   cudaGetErrorString(cudaGetLastError()));
    return fail(rc);
  }
  b->setup_ms = now_ms() - t0;
  *out = reinterpret_cast<bmg_batch*>(b);
  return BMG_OK;
}

static int batch_solve(bmg::Batch* b, const double* const* b_dev, double* const* x_dev, double tol,
                       bmg_info* per_prob, bmg_stream_t stream) {
  using namespace bmg;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const double t0 = now_ms();
  const bool pcg = b->opt.solver == BMG_SOLVER_PCG;
  std::vector<double*> user(2 * size_t(b->nprob));
  for (int p = 0; p < b->nprob; ++p) {
    user[p] = const_cast<double*>(b_dev[p]);
    user[b->nprob + p] = x_dev[p];
  }
  cudaMemcpyAsync(b->user, user.data(), sizeof(double*) * user.size(), cudaMemcpyHostToDevice, s);
  k_bpack<<<b->nunits, kKT, 0, s>>>(b->prob, b->units, b->user, b->nprob, pcg ? 1 : 0);
  count_launch();
  for (int p = 0; p < b->nprob; ++p) {
    Scalars z{};
    z.tol = tol;
    z.max_cycles = b->opt.max_cycles;
    b->sc_host[p] = z;
  }
  cudaMemcpyAsync(b->sc, b->sc_host, sizeof(Scalars) * b->nprob, cudaMemcpyHostToDevice, s);
  enqueue_residuals(b, 0, false, s);       // ||b||, go = (b != 0)
  if (pcg)
    enqueue_pcg_init(b, s);                // r = B - A X and the stop test
  else
    enqueue_residuals(b, 1, false, s);     // first residual and stop test
  if (cudaGraphLaunch(b->exec, s) != cudaSuccess) return BMG_ECUDA;
  k_bunpack<<<b->nunits, kKT, 0, s>>>(b->prob, b->units, b->sc, b->user, b->nprob, pcg ? 1 : 0);
  count_launch();
  if (cudaMemcpyAsync(b->sc_host, b->sc, sizeof(Scalars) * b->nprob, cudaMemcpyDeviceToHost, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return BMG_ECUDA;
  const double ms = now_ms() - t0;
  int rc = BMG_OK;
  for (int p = 0; p < b->nprob; ++p) {
    const Scalars& r = b->sc_host[p];
    if (per_prob) per_prob[p] = bmg_info{r.cycles, b->hs[p]->threshold, r.rel, b->setup_ms, ms, 1};
    if (r.err & DEV_NAN) rc = BMG_ENAN;
    else if ((r.err & DEV_TIMEOUT) && (rc == BMG_OK || rc == BMG_ENOCONV)) rc = BMG_ETIMEOUT;
    else if (!(r.rel <= tol) && r.bnorm2 > 0.0 && rc == BMG_OK) rc = BMG_ENOCONV;
  }
  return rc;
}

extern "C" int bmg_batch_solve(bmg_batch* bp, const double* const* b_dev, double* const* x_dev,
                               double tol, bmg_info* per_prob, bmg_stream_t stream) {
  Batch* b = reinterpret_cast<Batch*>(bp);
  if (!b || !b_dev || !x_dev || !(tol > 0.0)) return BMG_EINVAL;
  const int rc = batch_solve(b, b_dev, x_dev, tol, per_prob, stream);
  if (rc == BMG_ECUDA)
    for (bmg::Hierarchy* h : b->hs) h->pending.lost();
  return rc;
}

extern "C" void bmg_batch_destroy(bmg_batch* bp) { bmg::destroy_batch(reinterpret_cast<Batch*>(bp)); }

extern "C" int bmg_batch_size(const bmg_batch* bp, int* nprob) {
  const Batch* b = reinterpret_cast<const Batch*>(bp);
  if (!b || !nprob) return BMG_EINVAL;
  *nprob = b->nprob;
  return BMG_OK;
}
