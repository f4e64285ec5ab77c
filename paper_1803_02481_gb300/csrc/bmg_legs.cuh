// The two legs of a V-cycle level as one kernel each (Algorithm 1):
//   down: nu1 pre-smoothing sweeps, residual and restriction;
//   up:   interpolation and correction and one post-smoothing sweep, on the
//         finest level optionally with the next cycle's first colour work and
//         its stop test.
//
// Why.  Launched one operation at a time, a level of a few thousand points
// costs six launches of 2 to 5 us each (a chain of dependent FP64
// instructions at 64 cycles a step, the L2 round trip of its inputs, and the
// launch), and a level of millions of FP32 points moves the operator three
// times and the iterate and the residual several times more.  A block here
// stages the operator and b of its tile plus a halo once and takes every
// colour phase, the residual and the restriction from shared memory, so the
// level costs one L2 round trip and one launch per leg, and its planes cross
// the memory once per leg.
//
// How.  The redundant-halo scheme of the one-sweep kernels
// (bmg_sweep_tile.cuh), over all the leg's phases: phase g of G is relaxed on
// the tile grown by what the phases after it read, so no block needs another
// block's new values.  A block's halo points take the same operations on the
// same operands as their owner's, so every value is that of the separate
// kernels bit for bit.  The price is the halo's work: two four-colour sweeps
// grow the tile by 7 columns and 3 rows on each side.
//
// The down leg restricts at the coarse points inside its tile, which gather
// the residual one column and one row beyond it; the last sweep therefore
// covers the tile grown by one point below and two above.
//
// The up leg leaves out work whose result nothing reads: the post-smoothing
// sweep starts with the black points (5-point levels) or the coarse points
// (9-point levels), and replaces their values without reading them, so they
// are not interpolated.
#pragma once

#include "bmg_sweep_tile.cuh"

namespace bmg {

__device__ __forceinline__ void leg_copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   static_cast<unsigned>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void leg_copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

constexpr int round_up(int a, int b) { return (a + b - 1) / b * b; }
constexpr int max_int(int a, int b) { return a > b ? a : b; }

// A staged box: TX x TY tile, HA halo columns (a whole number of 16-byte
// units and even) and HY halo rows (even) on each side.
template <typename T, int TX, int TY, int NEEDX, int NEEDY>
struct LegBox {
  static constexpr int ALIGN = max_int(2, int(16 / sizeof(T)));
  static constexpr int HA = round_up(NEEDX, ALIGN), HY = round_up(NEEDY, 2);
  static constexpr int BW = TX + 2 * HA, BH = TY + 2 * HY, PL = BW * BH;
  static_assert(TX % ALIGN == 0 && TY % 2 == 0, "tiles keep alignment and colours");
};

template <typename T, bool NINE, int NS, int TX, int TY>
struct DownLeg {
  static constexpr int NPH = NINE ? 4 : 2, G = NS * NPH;
  static constexpr int grow_x(int g) { return G - 1 - g; }
  static constexpr int grow_y(int g) { return NINE ? 2 * NS - 1 - g / 2 : G - 1 - g; }
  using Box = LegBox<T, TX, TY, G + 2, (NINE ? 2 * NS : G) + 2>;
  static constexpr int NPL = NINE ? 8 : 6;   // x, b, 1/C, C, W, S (, SW, NW)
  static constexpr size_t SMEM = size_t(NPL) * Box::PL * sizeof(T);
};

template <typename T, bool NINE, int TX, int TY, bool NRM>
struct UpLeg {
  static constexpr int NPH = NINE ? 4 : 2, G = NPH + (NRM ? 1 : 0);
  static constexpr int grow_x(int g) { return G - 1 - g; }
  static constexpr int grow_y(int g) { return NINE ? 1 - g / 2 : G - 1 - g; }
  using Box = LegBox<T, TX, TY, G, NINE ? 2 : G>;
  static constexpr int NPL = NINE ? 7 : 5;   // x, b, 1/C, W, S (, SW, NW)
  static constexpr size_t SMEM = size_t(NPL) * Box::PL * sizeof(T);
};

enum LegPlane { LP_X = 0, LP_B, LP_IC, LP_W, LP_S, LP_C5, LP_SW = LP_C5, LP_NW, LP_C9 };

// Stages the box (first column i0 - HA, first row j0 - HY) of N planes, plane
// src[p] into slot[p]: the index arithmetic of a 16-byte unit serves all of
// them (plane by plane it cost 1.5 us of an 8.5 us leg).  Columns past the
// east ghost and rows outside the planes are left as they are: the points
// that would read them lie outside the grid and are not updated.
template <typename T, class Box, int NT, int N>
__device__ __forceinline__ void leg_stage(T* sm, const T* const (&src)[N], const int (&slot)[N], int i0,
                                          int j0, int nx, int ny, int pitch) {
  constexpr int PER = int(16 / sizeof(T)), CW = Box::BW / PER;
#pragma unroll 1
  for (int e = threadIdx.x; e < CW * Box::BH; e += NT) {
    const int r = e / CW, c = (e - r * CW) * PER;
    const int i = i0 - Box::HA + c, j = j0 - Box::HY + r;
    if (i <= nx + 1 && j >= 0 && j <= ny + 1) {
      T* d = sm + r * Box::BW + c;
      const ptrdiff_t o = ptrdiff_t(j) * pitch + i;
#pragma unroll
      for (int p = 0; p < N; ++p) leg_copy16(d + slot[p] * Box::PL, src[p] + o);
    }
  }
}

template <typename T, bool NINE, class Box>
__device__ __forceinline__ GsCoef<T, NINE> leg_coef(const T* sm, int o) {
  constexpr int PL = Box::PL, BW = Box::BW;
  GsCoef<T, NINE> c;
  c.b = sm[LP_B * PL + o];
  c.ic = sm[LP_IC * PL + o];
  c.w = sm[LP_W * PL + o];
  c.e = sm[LP_W * PL + o + 1];
  c.s = sm[LP_S * PL + o];
  c.n = sm[LP_S * PL + o + BW];
  if (NINE) {
    c.sw = sm[LP_SW * PL + o];
    c.se = sm[LP_NW * PL + o + 1 - BW];
    c.nw = sm[LP_NW * PL + o];
    c.ne = sm[LP_SW * PL + o + 1 + BW];
  }
  return c;
}

// The points of one colour phase on rows [r0, r1), columns [c0, c1) of the
// box: the sub-lattices in `colours` (one, or the two of a red-black colour:
// every second point of every row).  Point q's offset in the box, or -1
// outside the phase or the grid.
template <bool NINE, class Box>
__device__ __forceinline__ int leg_point(int q, int i0, int j0, int nx, int ny, unsigned colours, int r0,
                                         int r1, int c0, int c1) {
  // four colours: rows and columns of parity (pj, pi); red-black: every row,
  // columns of parity pi in even rows and 1 - pi in odd ones
  const int pj = NINE ? (colours >> 2 ? 1 : 0) : 0;
  const int pi = NINE ? (colours & 0xAu ? 1 : 0) : (colours & 1u ? 0 : 1);
  const int rf = NINE ? r0 + ((pj - r0) & 1) : r0, dr = NINE ? 2 : 1;
  const int nr = NINE ? (r1 - rf + 1) >> 1 : r1 - r0;
  const int cf = NINE ? c0 + ((pi - c0) & 1) : c0;
  const int ncol = (c1 - cf + 1) >> 1;
  const int rr = q / ncol, r = rf + dr * rr;
  int c = cf + 2 * (q - rr * ncol);
  if (!NINE) c += (pi + r + c0) & 1;
  const bool in = q < nr * ncol && c < c1 && unsigned(i0 + c - Box::HA - 1) < unsigned(nx) &&
                  unsigned(j0 + r - Box::HY - 1) < unsigned(ny);
  return in ? r * Box::BW + c : -1;
}
// Slots of a phase (an upper bound of q).
template <bool NINE>
__host__ __device__ constexpr int leg_points(int r0, int r1, int c0, int c1) {
  return (NINE ? (r1 - r0 + 1) / 2 : r1 - r0) * ((c1 - c0 + 1) / 2);
}

// G colour phases.  region(g) gives phase g's rows and columns, colours(g)
// its sub-lattices, terms(g) its neighbour terms; put(g, o, value) takes the
// new value of a point.  Every phase starts with a barrier.  A thread's first
// point of each phase is found beforehand, and its coefficients are loaded
// during the phase before (they are constant), so that a phase is the
// barrier, the loads of the iterate, the chain of its terms and a store.
struct LegRegion {
  int r0, r1, c0, c1;
};
template <typename T, bool NINE, class Box, int NT, int G, class R, class C, class M, class F>
__device__ __forceinline__ void leg_phases(T* sm, const int (&first)[G], int i0, int j0, int nx, int ny,
                                           R region, C colours, M terms, F put) {
  GsCoef<T, NINE> a, next;
  if (first[0] >= 0) a = leg_coef<T, NINE, Box>(sm, first[0]);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    __syncthreads();
    const LegRegion w = region(g);
    auto update = [&](const GsCoef<T, NINE>& cf, int o) {
      const T* xp = sm + o;   // LP_X
      put(g, o, gs_apply_masked<T, NINE>(cf, [&](int dx, int dy) { return xp[dx + dy * Box::BW]; }, terms(g)));
    };
    if (g + 1 < G && first[g + 1 < G ? g + 1 : g] >= 0)
      next = leg_coef<T, NINE, Box>(sm, first[g + 1 < G ? g + 1 : g]);
    if (first[g] >= 0) update(a, first[g]);
    const int n = leg_points<NINE>(w.r0, w.r1, w.c0, w.c1);
    for (int q = threadIdx.x + NT; q < n; q += NT) {
      const int o = leg_point<NINE, Box>(q, i0, j0, nx, ny, colours(g), w.r0, w.r1, w.c0, w.c1);
      if (o >= 0) update(leg_coef<T, NINE, Box>(sm, o), o);
    }
    a = next;
  }
}

// What a down leg may read before the kernel waits for its predecessor: the
// operator, and the restriction weights of the thread's coarse point.
template <typename T, bool NINE, int NS, int TX, int TY, int NT>
__device__ __forceinline__ void down_constants(const LevelV<T>& F, const LevelV<T>& Cc, T* sm, int bx,
                                               int by, T (&pw)[8]) {
  using Box = typename DownLeg<T, NINE, NS, TX, TY>::Box;
  static_assert((TX / 2) * (TY / 2) <= NT, "one coarse point per thread");
  const int i0 = bx * TX + 1, j0 = by * TY + 1;
  if constexpr (NINE) {
    const T* const src[] = {F.iC, F.W, F.S, F.SW, F.NW, F.C};
    const int slot[] = {LP_IC, LP_W, LP_S, LP_SW, LP_NW, LP_C9};
    leg_stage<T, Box, NT>(sm, src, slot, i0, j0, F.nx, F.ny, F.pitch);
  } else {
    const T* const src[] = {F.iC, F.W, F.S, F.C};
    const int slot[] = {LP_IC, LP_W, LP_S, LP_C5};
    leg_stage<T, Box, NT>(sm, src, slot, i0, j0, F.nx, F.ny, F.pitch);
  }
  // the iterate's box starts as zero (out-of-grid points stay so)
  static_assert(Box::PL * sizeof(T) % 16 == 0, "planes are whole 16-byte units");
  for (int e = threadIdx.x; e < int(Box::PL * sizeof(T) / 16); e += NT)
    reinterpret_cast<int4*>(sm + LP_X * Box::PL)[e] = make_int4(0, 0, 0, 0);
  const int dj = int(threadIdx.x) / (TX / 2), di = int(threadIdx.x) - dj * (TX / 2);
  const int I = bx * (TX / 2) + 1 + di, J = by * (TY / 2) + 1 + dj;
  if (dj < TY / 2 && I <= Cc.nx && J <= Cc.ny) {
    const int cp = Cc.pitch, c = J * cp + I;
    pw[0] = F.P[XE][c - 1];
    pw[1] = F.P[XW][c];
    pw[2] = F.P[YN][c - cp];
    pw[3] = F.P[YS][c];
    pw[4] = F.P[CNE][c - cp - 1];
    pw[5] = F.P[CNW][c - cp];
    pw[6] = F.P[CSE][c - 1];
    pw[7] = F.P[CSW][c];
  }
}

// The rest of the leg on tile (bx, by): reads the iterate from xin (ZERO: it
// is zero and not read), writes it to xout, and the restricted residual and a
// zero iterate to the coarse level Cc.
template <typename T, bool NINE, int NS, bool ZERO, int TX, int TY, int NT>
__device__ __forceinline__ void down_tile(const LevelV<T>& F, const T* __restrict__ xin,
                                          T* __restrict__ xout, const LevelV<T>& Cc, T* sm, int bx,
                                          int by, const T (&pw)[8]) {
  using D = DownLeg<T, NINE, NS, TX, TY>;
  using Box = typename D::Box;
  constexpr int BW = Box::BW, HA = Box::HA, HY = Box::HY, PL = Box::PL;
  const int nx = F.nx, ny = F.ny, i0 = bx * TX + 1, j0 = by * TY + 1;
  if constexpr (ZERO) {
    const T* const src[] = {F.b};
    const int slot[] = {LP_B};
    leg_stage<T, Box, NT>(sm, src, slot, i0, j0, nx, ny, F.pitch);
  } else {
    __syncthreads();   // the zeroed iterate, before its copies land
    const T* const src[] = {F.b, xin};
    const int slot[] = {LP_B, LP_X};
    leg_stage<T, Box, NT>(sm, src, slot, i0, j0, nx, ny, F.pitch);
  }
  auto region = [](int g) {
    const int gx = D::grow_x(g), gy = D::grow_y(g);
    return LegRegion{HY - 1 - gy, HY + TY + 2 + gy, HA - 1 - gx, HA + TX + 2 + gx};
  };
  auto colours = [](int g) {
    return ((NINE ? four_order(false) : rb_order(false)) >> (4 * (g % D::NPH))) & 0xFu;
  };
  auto terms = [](int g) { return ZERO && g < D::NPH ? zero_start_mask(NINE, g % D::NPH) : 0xFFu; };
  int first[D::G];
#pragma unroll
  for (int g = 0; g < D::G; ++g) {
    const LegRegion w = region(g);
    first[g] = leg_point<NINE, Box>(threadIdx.x, i0, j0, nx, ny, colours(g), w.r0, w.r1, w.c0, w.c1);
  }
  leg_copy_wait();
  __syncthreads();
  leg_phases<T, NINE, Box, NT, D::G>(sm, first, i0, j0, nx, ny, region, colours, terms,
                                     [&](int, int o, T v) { sm[o] = v; });
  __syncthreads();
  // the residual replaces b at its point; zero outside the grid
  const T* const sc = sm + (NINE ? LP_C9 : LP_C5) * PL;
  for (int e = threadIdx.x; e < (TX + 1) * (TY + 1); e += NT) {
    const int rr = e / (TX + 1), r = HY + rr, c = HA + e - rr * (TX + 1);
    const int o = r * BW + c;
    T v = T(0);
    if (i0 + c - HA <= nx && j0 + r - HY <= ny) {
      const GsCoef<T, NINE> a = leg_coef<T, NINE, Box>(sm, o);
      v = fma(-sc[o], sm[o], a.b);
      v = fma(a.w, sm[o - 1], v);
      v = fma(a.e, sm[o + 1], v);
      v = fma(a.s, sm[o - BW], v);
      v = fma(a.n, sm[o + BW], v);
      if (NINE) {
        v = fma(a.sw, sm[o - BW - 1], v);
        v = fma(a.se, sm[o - BW + 1], v);
        v = fma(a.nw, sm[o + BW - 1], v);
        v = fma(a.ne, sm[o + BW + 1], v);
      }
    }
    sm[LP_B * PL + o] = v;
  }
  for (int e = threadIdx.x; e < TX * TY; e += NT) {
    const int r = e / TX, c = e - r * TX;
    const int i = i0 + c, j = j0 + r;
    if (i <= nx && j <= ny) xout[ptrdiff_t(j) * F.pitch + i] = sm[(r + HY) * BW + c + HA];
  }
  __syncthreads();
  // coarse (I, J) is fine (2 I, 2 J): box row HY + 1 + 2 dj, column HA + 1 + 2 di
  // (the terms of restrict_value in its order)
  const int dj = int(threadIdx.x) / (TX / 2), di = int(threadIdx.x) - dj * (TX / 2);
  const int I = bx * (TX / 2) + 1 + di, J = by * (TY / 2) + 1 + dj;
  if (dj < TY / 2 && I <= Cc.nx && J <= Cc.ny) {
    const T* r = sm + LP_B * PL + (HY + 1 + 2 * dj) * BW + HA + 1 + 2 * di;
    T acc = r[0];
    acc = fma(pw[0], r[-1], acc);
    acc = fma(pw[1], r[1], acc);
    acc = fma(pw[2], r[-BW], acc);
    acc = fma(pw[3], r[BW], acc);
    acc = fma(pw[4], r[-BW - 1], acc);
    acc = fma(pw[5], r[-BW + 1], acc);
    acc = fma(pw[6], r[BW - 1], acc);
    acc = fma(pw[7], r[BW + 1], acc);
    Cc.b[J * Cc.pitch + I] = acc;
    Cc.x[J * Cc.pitch + I] = T(0);
  }
}

// The interpolation weights of the cell (fine points (2 I + 1, 2 J + 1) ..
// (2 I + 2, 2 J + 2)) that the leg uses: cell centre, and on 9-point levels
// the x-edge (2 I + 1, 2 J + 2) and the y-edge (2 I + 2, 2 J + 1).
template <typename T, bool NINE>
__device__ __forceinline__ void cell_weights(const LevelV<T>& F, int I, int J, bool in, T (&w)[8]) {
  if (!in) return;
  const int cp = F.cpitch, c = J * cp + I;
  w[0] = F.P[CSW][c];
  w[1] = F.P[CSE][c];
  w[2] = F.P[CNW][c];
  w[3] = F.P[CNE][c];
  if (NINE) {
    w[4] = F.P[XW][c + cp];
    w[5] = F.P[XE][c + cp];
    w[6] = F.P[YS][c + 1];
    w[7] = F.P[YN][c + 1];
  }
}

// What an up leg may read before the kernel waits for its predecessor: the
// operator, and the interpolation weights of the thread's first cell.
template <typename T, bool NINE, int TX, int TY, int NT, bool NRM>
__device__ __forceinline__ void up_constants(const LevelV<T>& F, T* sm, int bx, int by, T (&w)[8]) {
  using Box = typename UpLeg<T, NINE, TX, TY, NRM>::Box;
  const int i0 = bx * TX + 1, j0 = by * TY + 1;
  if constexpr (NINE) {
    const T* const src[] = {F.iC, F.W, F.S, F.SW, F.NW};
    const int slot[] = {LP_IC, LP_W, LP_S, LP_SW, LP_NW};
    leg_stage<T, Box, NT>(sm, src, slot, i0, j0, F.nx, F.ny, F.pitch);
  } else {
    const T* const src[] = {F.iC, F.W, F.S};
    const int slot[] = {LP_IC, LP_W, LP_S};
    leg_stage<T, Box, NT>(sm, src, slot, i0, j0, F.nx, F.ny, F.pitch);
  }
  const int rj = int(threadIdx.x) / (Box::BW / 2), ri = int(threadIdx.x) - rj * (Box::BW / 2);
  const int i = i0 - Box::HA + 2 * ri, j = j0 - Box::HY + 2 * rj;
  cell_weights<T, NINE>(F, i >> 1, j >> 1,
                        rj < Box::BH / 2 && i >= 1 && i <= F.nx && j >= 1 && j <= F.ny, w);
}

// x = xin + P xc and one reverse-order sweep on tile (bx, by), written to
// xout.  NRM (finest 5-point level): goes on with the next cycle's first
// pre-smoothing sweep, whose first phase would repeat the red values just
// written (see bmg_sweep_tma.cuh) and is left out; the black phase's
// C (x_new - x_old) is the residual of xout; its iterate goes to xnext and
// the block's sum of squares is returned (in thread 0).
template <typename T, bool NINE, int TX, int TY, int NT, bool NRM>
__device__ __forceinline__ double up_tile(const LevelV<T>& F, const T* __restrict__ xin,
                                          const T* __restrict__ xc, T* __restrict__ xout,
                                          T* __restrict__ xnext, T* sm, int bx, int by, T (&w)[8]) {
  static_assert(!(NRM && NINE), "the stop test is taken on the 5-point finest level");
  using U = UpLeg<T, NINE, TX, TY, NRM>;
  using Box = typename U::Box;
  constexpr int BW = Box::BW, BH = Box::BH, HA = Box::HA, HY = Box::HY;
  const int nx = F.nx, ny = F.ny, i0 = bx * TX + 1, j0 = by * TY + 1;
  {
    const T* const src[] = {F.b};
    const int slot[] = {LP_B};
    leg_stage<T, Box, NT>(sm, src, slot, i0, j0, nx, ny, F.pitch);
  }
  // the box's cells: interp_value's operations at the points that are read
  const int cp = F.cpitch;
  for (int e = threadIdx.x; e < (BW / 2) * (BH / 2); e += NT) {
    const int rj = e / (BW / 2), ri = e - rj * (BW / 2);
    const int i = i0 - HA + 2 * ri, j = j0 - HY + 2 * rj;   // odd
    const int I = i >> 1, J = j >> 1;
    const bool in = i >= 1 && i <= nx && j >= 1 && j <= ny;
    const bool e1 = in && i + 1 <= nx, n1 = in && j + 1 <= ny;
    if (e >= NT) cell_weights<T, NINE>(F, I, J, in, w);
    T c00 = 0, c10 = 0, c01 = 0, c11 = 0, x0 = 0, x1 = 0, x2 = 0;
    const ptrdiff_t o = ptrdiff_t(j) * F.pitch + i;
    if (in) {
      const T* q = xc + J * cp + I;
      c00 = q[0];
      c10 = q[1];
      c01 = q[cp];
      c11 = q[cp + 1];
      x0 = xin[o];
    }
    if (NINE) {
      if (n1) x1 = xin[o + F.pitch];
      if (e1) x2 = xin[o + 1];
    } else if (e1 && n1) {
      x1 = xin[o + F.pitch + 1];
    }
    T* xs = sm + (2 * rj) * BW + 2 * ri;
    T v = T(0);
    if (in) {
      v = w[0] * c00;
      v = fma(w[1], c10, v);
      v = fma(w[2], c01, v);
      v = fma(w[3], c11, v);
      v = x0 + v;
    }
    xs[0] = v;
    if (NINE) {
      xs[BW] = n1 ? x1 + fma(w[4], c01, w[5] * c11) : T(0);
      xs[1] = e1 ? x2 + fma(w[6], c10, w[7] * c11) : T(0);
      xs[BW + 1] = T(0);
    } else {
      xs[BW] = T(0);
      xs[1] = T(0);
      xs[BW + 1] = e1 && n1 ? x1 + c11 : T(0);
    }
  }
  // phase NPH (NRM) is the next cycle's black phase, on the tile alone
  auto region = [](int g) {
    const int gx = U::grow_x(g), gy = U::grow_y(g);
    return LegRegion{HY - gy, HY + TY + gy, HA - gx, HA + TX + gx};
  };
  auto colours = [](int g) {
    if (g == U::NPH) return (rb_order(false) >> 4) & 0xFu;
    return ((NINE ? four_order(true) : rb_order(true)) >> (4 * g)) & 0xFu;
  };
  int first[U::G];
#pragma unroll
  for (int g = 0; g < U::G; ++g) {
    const LegRegion w = region(g);
    first[g] = leg_point<NINE, Box>(threadIdx.x, i0, j0, nx, ny, colours(g), w.r0, w.r1, w.c0, w.c1);
  }
  auto write = [&](T* __restrict__ out, auto value) {
    for (int e = threadIdx.x; e < TX * TY; e += NT) {
      const int r = e / TX, c = e - r * TX;
      const int i = i0 + c, j = j0 + r;
      if (i <= nx && j <= ny) out[ptrdiff_t(j) * F.pitch + i] = value((r + HY) * BW + c + HA);
    }
  };
  leg_copy_wait();
  __syncthreads();
  // NRM: the residual's phase leaves the iterate as it is and puts the new
  // black values into b's plane, which no later phase reads
  double acc = 0.0;
  leg_phases<T, NINE, Box, NT, U::G>(
      sm, first, i0, j0, nx, ny, region, colours, [](int) { return 0xFFu; }, [&](int g, int o, T v) {
        if (NRM && g == U::NPH) {
          const int r = o / BW, c = o - r * BW;
          const double rv = double(F.C[ptrdiff_t(j0 + r - HY) * F.pitch + i0 + c - HA]) * double(v - sm[o]);
          acc = fma(rv, rv, acc);
          sm[LP_B * Box::PL + o] = v;
        } else {
          sm[o] = v;
        }
      });
  __syncthreads();
  write(xout, [&](int o) { return sm[o]; });
  if constexpr (NRM) {
    // red points (even sum of the box coordinates, as of the 0-based ones)
    // keep their values
    write(xnext, [&](int o) { return sm[((o / BW + o % BW) & 1) ? LP_B * Box::PL + o : o]; });
    // fixed reduction tree: warps, then warp sums in order
    __shared__ double wsum[NT / 32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = acc;
    __syncthreads();
    double a = 0.0;
    if (threadIdx.x == 0)
      for (int w = 0; w < NT / 32; ++w) a += wsum[w];
    return a;
  }
  return 0.0;
}

}  // namespace bmg
