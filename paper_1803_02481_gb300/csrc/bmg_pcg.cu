// Conjugate gradients on the finest operator, preconditioned by one
// symmetric V(nu, nu) cycle of Algorithm 1 from a zero initial guess (on the
// FP64 levels, or on the FP32 hierarchy of BMG_FP32_REFINE; an
// extension: the paper iterates V-cycles; with nu1 = nu2, the colours of the
// post-smoothing reversed, R = P^T and an exact coarsest solve, the cycle is
// a symmetric positive definite preconditioner).
//
// The vectors live on the finest FP64 level: the level's b plane holds the
// residual r (it is the V-cycle's right-hand side), its x plane z = M^{-1} r
// (the V-cycle's output), and Hierarchy::pcg_x, pcg_b, pcg_p, pcg_q hold the
// iterate, the right-hand side, the search direction and A p; with an FP32
// preconditioner z stays ||r|| times the FP32 iterate and no plane of its own.
// Every pass (bmg_krylov.cuh) walks the level with a fixed grid, fixed
// per-thread order and a fixed reduction tree (deterministic dot products);
// one thread then turns the partial sums into the scalars (alpha, beta, or
// the stop test of k_norm_final, which also drives the solve graph's WHILE
// node).  Measured on 16383 x 1023 with the FP32 preconditioner, per
// iteration: x and r 216 -> 119 us (48 B a point, 0.99 of the copy rate), r.z
// 156 -> 39 (with the former pass forming z), p 92 -> 68, the cast 69 -> 39.
#include "bmg_krylov.cuh"

#include <algorithm>

namespace bmg {

namespace {

template <int WHAT, bool F32>
__global__ void __launch_bounds__(kKT) k_pcg(LevelV<double> L, LevelV<float> F, PcgVec v,
                                             const Scalars* __restrict__ sc, int zero_z,
                                             double* __restrict__ partials) {
  griddep_wait();
  double s = krylov_pass<WHAT, F32>(L, &F, v, sc, zero_z != 0, blockIdx.x, gridDim.x);
  if (WHAT == K_P) return;
  s = krylov_block_sum(s);
  if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

__global__ void __launch_bounds__(kKT) k_pcg_cast(LevelV<double> L, LevelV<float> F,
                                                  const Scalars* __restrict__ sc, int zero_x) {
  griddep_wait();
  krylov_cast(L, F, sc, zero_x != 0, blockIdx.x, gridDim.x);
}

// One thread block sums the partials; what 0: rz = sum, beta = 0 (first
// direction); 1: alpha = rz / sum (sum = p.q); 2: beta = sum / rz, rz = sum
// (sum = r.z of the new residual).  e_only: the partials are of r.e with
// z = ||r|| e.  A zero denominator gives 0.
__global__ void __launch_bounds__(kKT) k_pcg_scalar(const double* __restrict__ partials, int n,
                                                    Scalars* sc, int what, int e_only) {
  griddep_wait();
  double acc = 0.0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) acc += partials[k];
  acc = krylov_block_sum(acc);
  if (threadIdx.x != 0) return;
  if (e_only) acc *= sc->rnorm;
  if (what == 0) {
    sc->rz = acc;
    sc->beta = 0.0;
  } else if (what == 1) {
    sc->alpha = acc != 0.0 ? sc->rz / acc : 0.0;
  } else {
    sc->beta = sc->rz != 0.0 ? acc / sc->rz : 0.0;
    sc->rz = acc;
  }
}

// Blocks of a pass: eight per SM (2048 threads), fewer on a smaller level.
int pass_blocks(const Hierarchy* h) {
  return std::min(pair_runs(h->nx, h->ny), std::min(8 * 152, h->max_partials));
}

bool fp32(const Hierarchy* h) { return h->opt.precision == BMG_FP32_REFINE; }

template <int WHAT>
int launch_pass(Hierarchy* h, cudaStream_t s) {
  const int nb = pass_blocks(h);
  const PcgVec v{h->pcg_x, h->pcg_b, h->pcg_p, h->pcg_q};
  const LevelV<float> F = fp32(h) ? h->f.back() : LevelV<float>{};
  const int zero_z = !fp32(h) && cycle_reads_zero_top(h);
  prof_begin(BMG_PROF_KRYLOV, s);
  if (fp32(h))
    launch_pdl(k_pcg<WHAT, true>, dim3(nb), dim3(kKT), 0, s, h->d.back(), F, v, (const Scalars*)h->sc,
               zero_z, h->partials);
  else
    launch_pdl(k_pcg<WHAT, false>, dim3(nb), dim3(kKT), 0, s, h->d.back(), F, v, (const Scalars*)h->sc,
               zero_z, h->partials);
  count_launch();
  return nb;
}

void launch_scalar(Hierarchy* h, int n, int what, cudaStream_t s) {
  launch_pdl(k_pcg_scalar, dim3(1), dim3(kKT), 0, s, (const double*)h->partials, n, h->sc, what,
             int(what != 1 && fp32(h)));
  count_launch();
}

}  // namespace

void launch_pcg_precond(Hierarchy* h, cudaStream_t s) {
  if (!fp32(h)) {
    enqueue_vcycle<double>(h, h->d, h->dlev64, h->threshold, s, -1, false, true);
    return;
  }
  launch_pdl(k_pcg_cast, dim3(pass_blocks(h)), dim3(kKT), 0, s, h->d.back(), h->f.back(),
             (const Scalars*)h->sc, int(cycle_reads_zero_top(h)));
  count_launch();
  enqueue_vcycle<float>(h, h->f, h->dlev32, h->threshold, s, -1, false, true);
}

void launch_pcg_init(Hierarchy* h, cudaStream_t s, bool in_graph) {
  const int n = launch_pass<K_INIT>(h, s);
  launch_norm_final(h, s, in_graph, n);
  prof_end(BMG_PROF_KRYLOV, s);
}

void launch_pcg_ap(Hierarchy* h, cudaStream_t s) {
  launch_scalar(h, launch_pass<K_AP>(h, s), 1, s);
  prof_end(BMG_PROF_KRYLOV, s);
}

void launch_pcg_xr(Hierarchy* h, cudaStream_t s, bool in_graph) {
  const int n = launch_pass<K_XR>(h, s);
  launch_norm_final(h, s, in_graph, n);
  prof_end(BMG_PROF_KRYLOV, s);
}

void launch_pcg_rz(Hierarchy* h, bool first, cudaStream_t s) {
  launch_scalar(h, launch_pass<K_RZ>(h, s), first ? 0 : 2, s);
  prof_end(BMG_PROF_KRYLOV, s);
}

void launch_pcg_p(Hierarchy* h, cudaStream_t s) {
  launch_pass<K_P>(h, s);
  prof_end(BMG_PROF_KRYLOV, s);
}

}  // namespace bmg
