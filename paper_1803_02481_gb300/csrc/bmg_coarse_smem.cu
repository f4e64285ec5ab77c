// The persistent coarse sub-cycle of one thread block with every plane of
// its levels in shared memory (Algorithm 1 on levels 0 .. thr-1, the
// single-GPU reading of the redistribution of Section 2.2 / Algorithm 2).
//
// What bounds it.  A sub-cycle on these few hundred points is a chain of
// short phases: per level nu1 + nu2 four-colour sweeps, residual,
// restriction and interpolation, each phase waiting for the one before.  On
// GB300 an FP64 instruction occupies its SM quarter for 64 cycles whatever
// the number of active lanes (measured: a dependent chain of fused
// multiply-adds runs at 64 cycles a step with one warp per quarter, and two
// independent chains in one warp take 128), so a phase of one warp per
// quarter cannot run faster than its nine terms, 580 cycles.  Loads from L2
// (296 cycles, measured) inside a phase come on top of that; a load from
// shared memory is 29 cycles and a barrier of 256 threads 29.  Hence:
//  * the constant planes of all levels are packed once at setup into one
//    image with the layout of shared memory, which one bulk copy brings in
//    before the kernel waits for its predecessor (a copy plane by plane spent
//    7 us on pointer loads and index arithmetic);
//  * a thread owns a 2 x 2 cell of a level, one point of each colour, and
//    holds its points' coefficients in registers over the sweeps and the
//    residual, so a phase is a barrier, eight loads of the iterate, the chain
//    and a store;
//  * the first sweep of a level, whose iterate is zero, applies only the
//    terms of the colours already updated.
//
// Every point is computed by the operations of gs_apply, resid_value,
// restrict_value and interp_value in their order, so the results are those
// of the other coarse kernels and of the full-grid launches bit for bit.
#include "bmg_internal.h"

#include <algorithm>

#include "bmg_sweep_tile.cuh"
#include "bmg_sweep_tma.cuh"

namespace bmg {

namespace {

constexpr int kNT = 256;          // two warps per SM quarter
constexpr int kMaxLevels = 12;    // levels a sub-cycle can hold
constexpr int kInvSmem = 96;      // the coarsest inverse is staged up to this size

// Constant planes of a level, each (nx + 2) x (ny + 2) elements with the
// zero ghost ring (5-point levels have no SW, NW), then its interpolation
// planes, (ncx + 1) x (ncy + 1) elements each.
enum { KC = 0, KIC, KW, KS, KSW, KNW, NK9 };
constexpr int kNK5 = KSW;

template <typename T>
struct SmArgs {
  int thr, nu1, nu2, add_rc;
  int top_nine;            // level thr - 1 is 9-point
  int top_zero;            // its iterate is zero on entry
  T *x, *b;                // its planes in global memory
  int pitch;
  CoarseSolve solve;       // the coarsest operator
  int inv_smem;            // its inverse is in the image
  int nx[kMaxLevels], ny[kMaxLevels];
  int koff[kMaxLevels];    // element offset of a level's constant planes
  int voff[kMaxLevels];    // element offset of its x, b (and r) planes
  int image_bytes;         // constants: planes, the inverse
  int foff;                // offset of the inverse in doubles
  int end;                 // end of the variable planes (elements)
  int soff;                // the coarsest right-hand side, in doubles
  const unsigned char* image;
  int* err;
};

template <typename T>
__device__ __forceinline__ T* shared_base() {
  extern __shared__ __align__(128) unsigned char sm_raw[];
  return reinterpret_cast<T*>(sm_raw);
}
// Element i of shared memory.
template <typename T>
__device__ __forceinline__ T& sh(int i) {
  return shared_base<T>()[i];
}

// A level's planes as element offsets into shared memory.
struct Lv {
  int nx, ny, sp, pl, x, b, r, k, P, pp, cp;
  template <typename T>
  __device__ __forceinline__ Lv(const SmArgs<T>& a, int l) {
    nx = a.nx[l];
    ny = a.ny[l];
    sp = nx + 2;
    pl = sp * (ny + 2);
    x = a.voff[l];
    b = x + pl;
    r = b + pl;
    k = a.koff[l];
    cp = l > 0 ? a.nx[l - 1] + 1 : 0;
    pp = l > 0 ? cp * (a.ny[l - 1] + 1) : 0;
    P = k + pl * (l == a.thr - 1 && !a.top_nine ? kNK5 : NK9);
  }
};

// A point's coefficients (b apart: it changes between the uses).
template <typename T>
struct Coef {
  T ic, c, w, e, s, n, sw, se, nw, ne;
};

template <typename T, bool NINE>
__device__ __forceinline__ void load_coef(Coef<T>& c, const Lv& L, int o) {
  const int q = L.k + o;
  c.c = sh<T>(q + KC * L.pl);
  c.ic = sh<T>(q + KIC * L.pl);
  c.w = sh<T>(q + KW * L.pl);
  c.e = sh<T>(q + KW * L.pl + 1);
  c.s = sh<T>(q + KS * L.pl);
  c.n = sh<T>(q + KS * L.pl + L.sp);
  if (NINE) {
    c.sw = sh<T>(q + KSW * L.pl);
    c.se = sh<T>(q + KNW * L.pl + 1 - L.sp);
    c.nw = sh<T>(q + KNW * L.pl);
    c.ne = sh<T>(q + KSW * L.pl + 1 + L.sp);
  }
}

// gs_apply_masked at shared offset o of the iterate.
template <typename T, bool NINE>
__device__ __forceinline__ T gauss_seidel(const Coef<T>& c, T b, int o, int sp, unsigned mask) {
  T acc = b;
  if (mask & 0x01u) acc = fma(c.w, sh<T>(o - 1), acc);
  if (mask & 0x02u) acc = fma(c.e, sh<T>(o + 1), acc);
  if (mask & 0x04u) acc = fma(c.s, sh<T>(o - sp), acc);
  if (mask & 0x08u) acc = fma(c.n, sh<T>(o + sp), acc);
  if (NINE) {
    if (mask & 0x10u) acc = fma(c.sw, sh<T>(o - sp - 1), acc);
    if (mask & 0x20u) acc = fma(c.se, sh<T>(o - sp + 1), acc);
    if (mask & 0x40u) acc = fma(c.nw, sh<T>(o + sp - 1), acc);
    if (mask & 0x80u) acc = fma(c.ne, sh<T>(o + sp + 1), acc);
  }
  return acc * c.ic;
}

// resid_value at shared offset o of the iterate.
template <typename T, bool NINE>
__device__ __forceinline__ T residual(const Coef<T>& c, T b, int o, int sp) {
  T r = fma(-c.c, sh<T>(o), b);
  r = fma(c.w, sh<T>(o - 1), r);
  r = fma(c.e, sh<T>(o + 1), r);
  r = fma(c.s, sh<T>(o - sp), r);
  r = fma(c.n, sh<T>(o + sp), r);
  if (NINE) {
    r = fma(c.sw, sh<T>(o - sp - 1), r);
    r = fma(c.se, sh<T>(o - sp + 1), r);
    r = fma(c.nw, sh<T>(o + sp - 1), r);
    r = fma(c.ne, sh<T>(o + sp + 1), r);
  }
  return r;
}

// A thread's 2 x 2 cell: point q = 2 pj + pi has 0-based parities (pj, pi).
template <typename T>
struct Cell {
  Coef<T> c[4];
  T b[4];
  int o;          // plane offset of point 0
  bool in[4];
};

template <typename T, bool NINE>
__device__ __forceinline__ void load_cell(Cell<T>& q, const Lv& L, int t) {
  const int hx = (L.nx + 1) >> 1;
  const int jj = t / hx, ii = t - jj * hx;
  q.o = (1 + 2 * jj) * L.sp + 1 + 2 * ii;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    q.in[k] = 2 * ii + (k & 1) < L.nx && 2 * jj + (k >> 1) < L.ny;
    const int o = q.o + (k >> 1) * L.sp + (k & 1);
    if (q.in[k]) {
      load_coef<T, NINE>(q.c[k], L, o);
      q.b[k] = sh<T>(L.b + o);
    }
  }
}

// The cells' coefficients kept over the whole sub-cycle: every level has
// threads of its own (`own`: this thread's level is the one at work), so they
// are loaded once, before the kernel waits for its predecessor, instead of in
// each leg of each level (500 ns a time).  Colour phase c.
template <typename T, bool NINE>
__device__ __forceinline__ void colour_own(const Cell<T>& q, const Lv& L, bool own, int c, unsigned mask) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (NINE ? k != c : ((k >> 1) ^ (k & 1)) != c) continue;
    if (own && q.in[k]) {
      const int d = q.o + (k >> 1) * L.sp + (k & 1);
      const int o = L.x + d;
      sh<T>(o) = gauss_seidel<T, NINE>(q.c[k], sh<T>(L.b + d), o, L.sp, mask);
    }
  }
  __syncthreads();
}

// Colour phase c (0 .. 3, or red 0 and black 1) on the cells of the block:
// `held` is the thread's own cell (of the first kNT); levels with more cells
// load the others' coefficients in the phase.
template <typename T, bool NINE>
__device__ __forceinline__ void colour(const Cell<T>& held, const Lv& L, int ncell, int c,
                                       unsigned mask) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (NINE ? k != c : ((k >> 1) ^ (k & 1)) != c) continue;
    const int d = (k >> 1) * L.sp + (k & 1);
    if (held.in[k]) {
      const int o = L.x + held.o + d;
      sh<T>(o) = gauss_seidel<T, NINE>(held.c[k], held.b[k], o, L.sp, mask);
    }
    for (int t = int(threadIdx.x) + kNT; t < ncell; t += kNT) {
      const int hx = (L.nx + 1) >> 1;
      const int jj = t / hx, ii = t - jj * hx;
      if (2 * ii + (k & 1) >= L.nx || 2 * jj + (k >> 1) >= L.ny) continue;
      const int o = (1 + 2 * jj) * L.sp + 1 + 2 * ii + d;
      Coef<T> cf;
      load_coef<T, NINE>(cf, L, o);
      sh<T>(L.x + o) = gauss_seidel<T, NINE>(cf, sh<T>(L.b + o), L.x + o, L.sp, mask);
    }
  }
  __syncthreads();
}

template <typename T, bool NINE, bool REVERSE, bool OWN>
__device__ __forceinline__ void sweep(const Cell<T>& held, const Lv& L, bool own, int ncell) {
  constexpr int NC = NINE ? 4 : 2;
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    const int c = REVERSE ? NC - 1 - k : k;
    if (OWN)
      colour_own<T, NINE>(held, L, own, c, NINE ? 0xFFu : 0x0Fu);
    else
      colour<T, NINE>(held, L, ncell, c, NINE ? 0xFFu : 0x0Fu);
  }
}

// Pre-smoothing, residual and restriction of a level.  Enters and leaves
// with every thread's writes visible.
template <typename T, bool NINE, bool OWN>
__device__ __forceinline__ void down(const Lv& L, const Lv& C, Cell<T>& held, bool own, int nu1, bool zero) {
  const int ncell = ((L.nx + 1) >> 1) * ((L.ny + 1) >> 1);
  if (!OWN) {
    held = Cell<T>{};
    if (int(threadIdx.x) < ncell) load_cell<T, NINE>(held, L, threadIdx.x);
  }
  int s = 0;
  if (zero && nu1 > 0) {
    constexpr int NC = NINE ? 4 : 2;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      if (OWN)
        colour_own<T, NINE>(held, L, own, k, zero_start_mask(NINE, k));
      else
        colour<T, NINE>(held, L, ncell, k, zero_start_mask(NINE, k));
    }
    s = 1;
  }
  for (; s < nu1; ++s) sweep<T, NINE, false, OWN>(held, L, own, ncell);
  if (OWN || 4 * ncell <= kNT) {
    // one point per thread, over all warps, instead of four in a few
    const int k = int(threadIdx.x) / (kNT / 4);
    const int hx = (L.nx + 1) >> 1;
    for (int t = int(threadIdx.x) % (kNT / 4); t < ncell; t += kNT / 4) {
      const int jj = t / hx, ii = t - jj * hx;
      if (2 * ii + (k & 1) >= L.nx || 2 * jj + (k >> 1) >= L.ny) continue;
      const int o = (1 + 2 * jj + (k >> 1)) * L.sp + 1 + 2 * ii + (k & 1);
      Coef<T> cf;
      load_coef<T, NINE>(cf, L, o);
      sh<T>(L.r + o) = residual<T, NINE>(cf, sh<T>(L.b + o), L.x + o, L.sp);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int d = (k >> 1) * L.sp + (k & 1);
      if (held.in[k])
        sh<T>(L.r + held.o + d) = residual<T, NINE>(held.c[k], held.b[k], L.x + held.o + d, L.sp);
    }
  }
  for (int t = int(threadIdx.x) + kNT; !OWN && t < ncell; t += kNT) {
    const int hx = (L.nx + 1) >> 1;
    const int jj = t / hx, ii = t - jj * hx;
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
      if (2 * ii + (k & 1) >= L.nx || 2 * jj + (k >> 1) >= L.ny) continue;
      const int o = (1 + 2 * jj + (k >> 1)) * L.sp + 1 + 2 * ii + (k & 1);
      Coef<T> cf;
      load_coef<T, NINE>(cf, L, o);
      sh<T>(L.r + o) = residual<T, NINE>(cf, sh<T>(L.b + o), L.x + o, L.sp);
    }
  }
  // restriction: the weights do not wait for the residual
  int J = int(threadIdx.x) / C.nx, I = int(threadIdx.x) - J * C.nx;
  for (int t = threadIdx.x; t - int(threadIdx.x) < C.nx * C.ny; t += kNT) {
    const bool in = t < C.nx * C.ny;
    if (t >= kNT) {
      J = t / C.nx;
      I = t - J * C.nx;
    }
    const int c = L.P + (J + 1) * L.cp + I + 1;
    T w[8];
    if (in) {
      w[0] = sh<T>(c + XE * L.pp - 1);
      w[1] = sh<T>(c + XW * L.pp);
      w[2] = sh<T>(c + YN * L.pp - L.cp);
      w[3] = sh<T>(c + YS * L.pp);
      w[4] = sh<T>(c + CNE * L.pp - L.cp - 1);
      w[5] = sh<T>(c + CNW * L.pp - L.cp);
      w[6] = sh<T>(c + CSE * L.pp - 1);
      w[7] = sh<T>(c + CSW * L.pp);
    }
    if (t < kNT) __syncthreads();   // (once, by every thread)
    if (in) {
      const int f = L.r + (2 * J + 2) * L.sp + 2 * I + 2;
      T acc = sh<T>(f);
      acc = fma(w[0], sh<T>(f - 1), acc);
      acc = fma(w[1], sh<T>(f + 1), acc);
      acc = fma(w[2], sh<T>(f - L.sp), acc);
      acc = fma(w[3], sh<T>(f + L.sp), acc);
      acc = fma(w[4], sh<T>(f - L.sp - 1), acc);
      acc = fma(w[5], sh<T>(f - L.sp + 1), acc);
      acc = fma(w[6], sh<T>(f + L.sp - 1), acc);
      acc = fma(w[7], sh<T>(f + L.sp + 1), acc);
      sh<T>(C.b + (J + 1) * C.sp + I + 1) = acc;
    }
  }
  __syncthreads();
}

// x += P x_c.  A fine point's work depends on its kind (cell centre, x-edge,
// y-edge, coarse point), and an FP64 instruction costs a full issue slot
// however few lanes take it: the kinds go to threads kNT / 4 apart, so that
// a warp holds one kind.  skip_coarse: a reverse-order sweep follows on a
// 9-point level, whose first phase replaces the coarse points without
// reading them.
template <typename T>
__device__ __forceinline__ void interpolate(const Lv& L, const Lv& C, bool add_rc, bool skip_coarse) {
  constexpr int G = kNT / 4;
  const int kind = int(threadIdx.x) / G;
  if (kind == 3 && skip_coarse) return;
  const int w = ((L.nx - 1) >> 1) + 1, n = w * (((L.ny - 1) >> 1) + 1);
  const int dx = kind < 2 ? 1 : 2;                 // centre, x-edge: odd column
  const int dy = kind == 0 || kind == 2 ? 1 : 2;   // centre, y-edge: odd row
  const int t0 = int(threadIdx.x) - kind * G;
  int J = t0 / w, I = t0 - J * w;
  const int dJ = G / w, dI = G - dJ * w;
  for (int t = t0; t < n; t += G) {
    const int i = 2 * I + dx, j = 2 * J + dy;
    if (i <= L.nx && j <= L.ny) {
      const int o = j * L.sp + i;
      const int ci = i >> 1, cj = j >> 1;
      const int c = L.P + cj * L.cp + ci, xc = C.x + cj * C.sp + ci;
      T v;
      if (kind == 0) {
        v = sh<T>(c + CSW * L.pp) * sh<T>(xc);
        v = fma(sh<T>(c + CSE * L.pp), sh<T>(xc + 1), v);
        v = fma(sh<T>(c + CNW * L.pp), sh<T>(xc + C.sp), v);
        v = fma(sh<T>(c + CNE * L.pp), sh<T>(xc + C.sp + 1), v);
      } else if (kind == 1) {
        v = fma(sh<T>(c + XW * L.pp), sh<T>(xc), sh<T>(c + XE * L.pp) * sh<T>(xc + 1));
      } else if (kind == 2) {
        v = fma(sh<T>(c + YS * L.pp), sh<T>(xc), sh<T>(c + YN * L.pp) * sh<T>(xc + C.sp));
      } else {
        v = sh<T>(xc);
      }
      if (add_rc && kind != 3) v = fma(sh<T>(L.r + o), sh<T>(L.k + KIC * L.pl + o), v);
      sh<T>(L.x + o) = sh<T>(L.x + o) + v;
    }
    I += dI;
    J += dJ;
    if (I >= w) {
      I -= w;
      ++J;
    }
  }
}

template <typename T, bool NINE, bool OWN>
__device__ __forceinline__ void up(const Lv& L, const Lv& C, Cell<T>& held, bool own, int nu2, bool add_rc) {
  const int ncell = ((L.nx + 1) >> 1) * ((L.ny + 1) >> 1);
  if (!OWN) {
    held = Cell<T>{};
    if (nu2 > 0 && int(threadIdx.x) < ncell) load_cell<T, NINE>(held, L, threadIdx.x);
  }
  interpolate<T>(L, C, add_rc, NINE && nu2 > 0);
  __syncthreads();
  for (int s = 0; s < nu2; ++s) sweep<T, NINE, true, OWN>(held, L, own, ncell);
}

// x_0 = A_0^{-1} b_0 with the stored inverse (the sums of blk_coarse_solve):
// one unknown per thread, or above kInverseSerial unknowns four lanes for
// each, one partial sum a lane; or by substitution.
template <typename T>
__device__ __forceinline__ void solve0(const SmArgs<T>& a, const Lv& L) {
  const int n = a.solve.n, nx = L.nx;
  if (!a.solve.product) {
    substitute(a.solve, &sh<double>(a.soff));
    for (int r = threadIdx.x; r < n; r += kNT)
      sh<T>(L.x + (r / nx + 1) * L.sp + r % nx + 1) = T(sh<double>(a.soff + r));
    return;
  }
  const bool quad = n > kInverseSerial;
  const int per = quad ? 4 : 1, k = quad ? int(threadIdx.x) & 3 : 0;
  for (int r0 = 0; r0 < n; r0 += kNT / per) {
    const int r = r0 + int(threadIdx.x) / per;
    if (r0 + (int(threadIdx.x) & ~31) / per >= n) break;   // (warp-uniform)
    const int q = r < n ? r : 0;
    auto inv = [&](int c) {
      return a.inv_smem ? sh<double>(a.foff + c * n + q) : a.solve.inv[size_t(c) * n + q];
    };
    auto b = [&](int c) { return sh<double>(a.soff + c); };
    double x = inverse_part(n, k, per, inv, b);
    if (quad) {
      x += __shfl_xor_sync(0xffffffffu, x, 1);
      x += __shfl_xor_sync(0xffffffffu, x, 2);
    }
    if (k == 0 && r < n) sh<T>(L.x + (r / nx + 1) * L.sp + r % nx + 1) = T(x);
  }
}

template <typename T, bool OWN>
__device__ __forceinline__ void coarse_smem_body(const SmArgs<T>& a) {
  using namespace tma_detail;
  __shared__ __align__(8) uint64_t bar;
  const int top = a.thr - 1;
  // no level above the coarsest here and an inverse too large to stage: the
  // image is empty, and a bulk copy of no bytes is not defined
  const bool staged = a.image_bytes > 0;
  if (staged && threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
    mbar_expect_tx(&bar, unsigned(a.image_bytes));
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
            saddr(shared_base<unsigned char>())),
        "l"(a.image), "r"(a.image_bytes), "r"(saddr(&bar))
        : "memory");
  }
  // zero iterates (with their ghosts) and the residuals' ghosts, which the
  // restriction of an even side reads
  for (int e = a.voff[0] + threadIdx.x; e < a.end; e += kNT) sh<T>(e) = T(0);
  __syncthreads();
  Cell<T> held{};
  int mine = 0;                          // OWN: this thread's level
  bool ok = true;
  if (OWN) {
    // levels top .. 1 take warps in turn
    if (staged) ok = mbar_wait_bounded(&bar, 0);
    int first = 0;
    for (int l = top; ok && l >= 1; --l) {
      const Lv L(a, l);
      const int n = ((L.nx + 1) >> 1) * ((L.ny + 1) >> 1), t = int(threadIdx.x) - first;
      if (t >= 0 && t < n) {
        mine = l;
        if (l < top || a.top_nine)
          load_cell<T, true>(held, L, t);
        else
          load_cell<T, false>(held, L, t);
      }
      first += (n + 31) & ~31;
    }
  }
  griddep_wait();
  griddep_launch();
  {
    const Lv L(a, top);
    const int w = L.nx;
    for (int t = threadIdx.x; t < w * L.ny; t += kNT) {
      const int j = t / w + 1, i = t - (j - 1) * w + 1;
      sh<T>(L.b + j * L.sp + i) = a.b[j * a.pitch + i];
      if (!a.top_zero) sh<T>(L.x + j * L.sp + i) = a.x[j * a.pitch + i];
    }
  }
  if (!OWN && staged) ok = mbar_wait_bounded(&bar, 0);
  if (!__syncthreads_and(ok)) {
    if (threadIdx.x == 0) {
      atomicOr(a.err, DEV_TIMEOUT);
      mbar_wait_bounded(&bar, 0);   // shared memory must outlive the copy
    }
    __syncthreads();
    return;
  }
  for (int l = top; l >= 1; --l) {
    const Lv L(a, l), C(a, l - 1);
    const bool zero = l < top || a.top_zero;
    if (l < top || a.top_nine)
      down<T, true, OWN>(L, C, held, mine == l, a.nu1, zero);
    else
      down<T, false, OWN>(L, C, held, mine == l, a.nu1, zero);
  }
  {
    const Lv L(a, 0);
    for (int r = threadIdx.x; r < a.solve.n; r += kNT)
      sh<double>(a.soff + r) = double(sh<T>(L.b + (r / L.nx + 1) * L.sp + r % L.nx + 1));
    __syncthreads();
    solve0<T>(a, L);
  }
  __syncthreads();
  for (int l = 1; l <= top; ++l) {
    const Lv L(a, l), C(a, l - 1);
    if (l < top || a.top_nine)
      up<T, true, OWN>(L, C, held, mine == l, a.nu2, a.add_rc != 0);
    else
      up<T, false, OWN>(L, C, held, mine == l, a.nu2, a.add_rc != 0);
    if (a.nu2 == 0) __syncthreads();
  }
  const Lv L(a, top);
  for (int t = threadIdx.x; t < L.nx * L.ny; t += kNT) {
    const int j = t / L.nx + 1, i = t - (j - 1) * L.nx + 1;
    a.x[j * a.pitch + i] = sh<T>(L.x + j * L.sp + i);
  }
}

template <typename T, bool OWN>
__global__ void __launch_bounds__(kNT, 1) k_coarse_smem(const __grid_constant__ SmArgs<T> a) {
  coarse_smem_body<T, OWN>(a);
}

// One problem per block; a problem that has stopped is left alone.  (`go` was
// settled before the kernel that precedes this one began.)
__global__ void __launch_bounds__(kNT, 1) k_coarse_smem_batch(const SmArgs<float>* __restrict__ args,
                                                             const Scalars* __restrict__ sc) {
  __shared__ SmArgs<float> a;
  if (!sc[blockIdx.x].go) {
    griddep_wait();   // (the kernel that follows relies on it)
    return;
  }
  const int* src = reinterpret_cast<const int*>(args + blockIdx.x);
  for (int e = threadIdx.x; e < int(sizeof(a) / sizeof(int)); e += kNT) reinterpret_cast<int*>(&a)[e] = src[e];
  __syncthreads();
  coarse_smem_body<float, false>(a);
}

// The image: blockIdx.x walks the constant planes of the levels (NK9 + NPW
// slots each), the last block the coarsest inverse.
template <typename T>
__global__ void k_coarse_image(const __grid_constant__ SmArgs<T> a, const LevelV<T>* lev,
                               unsigned char* image) {
  if (blockIdx.x == gridDim.x - 1) {
    double* d = reinterpret_cast<double*>(image) + a.foff;
    if (a.inv_smem)
      for (int e = threadIdx.x; e < a.solve.n * a.solve.n; e += blockDim.x) d[e] = a.solve.inv[e];
    return;
  }
  const int l = 1 + blockIdx.x / (NK9 + NPW), p = blockIdx.x % (NK9 + NPW);
  const Lv V(a, l);
  const LevelV<T>& L = lev[l];
  T* out = reinterpret_cast<T*>(image);
  if (p < NK9) {
    const T* src = p == KC ? L.C : p == KIC ? L.iC : p == KW ? L.W : p == KS ? L.S : p == KSW ? L.SW : L.NW;
    if (!src) return;
    for (int e = threadIdx.x; e < V.pl; e += blockDim.x) {
      const int j = e / V.sp, i = e - j * V.sp;
      out[V.k + p * V.pl + e] = src[size_t(j) * L.pitch + i];
    }
  } else {
    const T* src = L.P[p - NK9];
    for (int e = threadIdx.x; e < V.pp; e += blockDim.x) {
      const int j = e / V.cp, i = e - j * V.cp;
      out[V.P + (p - NK9) * V.pp + e] = src[size_t(j) * L.cpitch + i];
    }
  }
}

// Fills the layout of levels 0 .. thr-1; returns the shared memory it takes
// (0: it does not apply).
template <typename T>
size_t layout(const Hierarchy* h, int thr, SmArgs<T>& a) {
  if (thr < 1 || thr > kMaxLevels || thr > h->L || h->opt.smoother != BMG_SMOOTH_POINT) return 0;
  size_t off = 0;
  for (int l = 1; l < thr; ++l) {
    const Geom& g = h->geo64[l];
    const size_t pl = size_t(g.nx + 2) * (g.ny + 2);
    if (pl > kCoarseImageMax / sizeof(T)) return 0;
    a.koff[l] = int(off);
    off += pl * (l != h->L - 1 ? NK9 : kNK5);
    off += size_t(NPW) * (h->geo64[l - 1].nx + 1) * (h->geo64[l - 1].ny + 1);
    if (off * sizeof(T) > kCoarseImageMax) return 0;
  }
  const size_t n0 = size_t(h->n0);
  a.inv_smem = n0 <= kInvSmem;
  a.foff = int((off * sizeof(T) + 7) / 8);
  size_t bytes = 8 * (size_t(a.foff) + (a.inv_smem ? n0 * n0 : 0));
  bytes = (bytes + 15) / 16 * 16;
  a.image_bytes = int(bytes);
  off = bytes / sizeof(T);
  for (int l = 0; l < thr; ++l) {
    const Geom& g = h->geo64[l];
    a.nx[l] = g.nx;
    a.ny[l] = g.ny;
    a.voff[l] = int(off);
    off += size_t(g.nx + 2) * (g.ny + 2) * (l == 0 ? 2 : 3);
    if (off * sizeof(T) > kCoarseImageMax) return 0;
  }
  a.end = int(off);
  a.soff = int((off * sizeof(T) + 7) / 8);
  bytes = 8 * (size_t(a.soff) + n0);
  a.thr = thr;
  a.top_nine = thr < h->L;
  a.nu1 = h->opt.nu1;
  a.nu2 = h->opt.nu2;
  a.add_rc = h->opt.interp_residual_term;
  a.solve = coarse_solve(h);
  a.image = h->coarse_image;
  a.err = &h->sc->err;
  return bytes <= kCoarseImageMax ? bytes : 0;
}

template <typename T>
bool prepare() {
  return use_shared(k_coarse_smem<T, true>, kCoarseImageMax) && use_shared(k_coarse_smem<T, false>, kCoarseImageMax);
}

template <typename T>
int build_image(Hierarchy* h, const LevelV<T>* lev, cudaStream_t s) {
  SmArgs<T> a{};
  if (!layout<T>(h, h->threshold, a)) return BMG_ECUDA;
  k_coarse_image<T><<<(h->threshold - 1) * (NK9 + NPW) + 1, 256, 0, s>>>(a, lev,
                                                                         h->coarse_image);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? BMG_OK : BMG_ECUDA;
}

}  // namespace

bool coarse_smem_fits(const Hierarchy* h, int thr) {
  // (a prescaled finest level never fits: it is at least 1024 points wide)
  if (thr == h->L && h->opt.precision != BMG_FP32_REFINE && h->d.back().PR[PR_B]) return false;
  if (h->opt.precision == BMG_FP32_REFINE) {
    SmArgs<float> a{};
    return layout<float>(h, thr, a) > 0 && prepare<float>();
  }
  SmArgs<double> a{};
  return layout<double>(h, thr, a) > 0 && prepare<double>();
}

int launch_coarse_image(Hierarchy* h, cudaStream_t s) {
  if (!h->coarse_smem) return BMG_OK;
  return h->opt.precision == BMG_FP32_REFINE ? build_image<float>(h, h->dlev32, s)
                                             : build_image<double>(h, h->dlev64, s);
}

// The levels below h->threshold, or (a cycle that starts on a coarser level)
// fewer of them: the image of the first thr levels is a prefix of the whole
// but for the inverse, so the image of h->threshold levels is brought in.
template <typename T>
void launch_coarse_smem(Hierarchy* h, const LevelV<T>& top, int thr, bool top_zero, cudaStream_t s) {
  SmArgs<T> a{};
  const size_t bytes = layout<T>(h, h->threshold, a);
  a.thr = thr;
  a.top_nine = thr < h->L;
  a.top_zero = top_zero;
  a.x = top.x;
  a.b = top.b;
  a.pitch = top.pitch;
  // threads of its own for every level, where the block has as many
  int threads = 0;
  for (int l = 1; l < thr; ++l) threads += (((a.nx[l] + 1) / 2) * ((a.ny[l] + 1) / 2) + 31) / 32 * 32;
  if (threads <= kNT)
    launch_pdl(k_coarse_smem<T, true>, dim3(1), dim3(kNT), bytes, s, a);
  else
    launch_pdl(k_coarse_smem<T, false>, dim3(1), dim3(kNT), bytes, s, a);
}

size_t coarse_smem_batch_args(const Hierarchy* h, int* err, std::vector<unsigned char>& out) {
  static_assert(sizeof(SmArgs<float>) % sizeof(int) == 0, "copied by words");
  SmArgs<float> a{};
  const size_t bytes = layout<float>(h, h->threshold, a);
  const LevelV<float>& top = h->f[h->threshold - 1];
  a.top_zero = 1;
  a.add_rc = 0;   // (the batch leaves the r/C term out on every level)
  a.err = err;
  a.x = top.x;
  a.b = top.b;
  a.pitch = top.pitch;
  const unsigned char* p = reinterpret_cast<const unsigned char*>(&a);
  out.insert(out.end(), p, p + sizeof(a));
  return bytes;
}

bool coarse_smem_batch_ready() { return use_shared(k_coarse_smem_batch, kCoarseImageMax); }

void launch_coarse_smem_batch(const void* args, int count, size_t bytes, const Scalars* sc, cudaStream_t s) {
  launch_pdl(k_coarse_smem_batch, dim3(unsigned(count)), dim3(kNT), bytes, s,
             static_cast<const SmArgs<float>*>(args), sc);
  count_launch();
}

template void launch_coarse_smem<double>(Hierarchy*, const LevelV<double>&, int, bool, cudaStream_t);
template void launch_coarse_smem<float>(Hierarchy*, const LevelV<float>&, int, bool, cudaStream_t);

}  // namespace bmg
