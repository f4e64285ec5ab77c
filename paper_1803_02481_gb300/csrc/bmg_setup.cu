// BoxMG setup kernels (Section 2; discretisation of Section 5):
//   assembly of the 5-point cell-centred FV operator, operator-induced
//   interpolation weights, the Galerkin product P^T A P, the Cholesky factor
//   of the coarsest operator, dense <-> plane copies, and the backward of the
//   assembly (adjoint gradient).
#include "bmg_divide.cuh"
#include "bmg_internal.h"

#include <cmath>

namespace bmg {

namespace {

constexpr int kTB = 256;

inline int cdiv(long a, long b) { return int((a + b - 1) / b); }

// Face coefficient of two square cells (series conductance of the two half
// cells, Section 5 discretisation): 2 k1 k2 / (k1 + k2).
__device__ __forceinline__ double harmonic(double k1, double k2) {
  return 2.0 * k1 * k2 / (k1 + k2);
}

// k of cell q: the input itself, or exp(input) for log-coefficients.
__device__ __forceinline__ double cell_k(const double* __restrict__ k, size_t q, bool log_k) {
  return log_k ? exp(k[q]) : k[q];
}

// Tile of the assembly (cells) and of the weights (coarse indices): one thread
// each.
constexpr int kAX = 32, kAY = 8;

// Face and cell factors of the assembly: D = diag(k / r, k r) on cells of
// aspect hy / hx.  x faces carry harmonic(k_1 / r, k_2 / r) * hy / hx, y
// faces harmonic(k_1 r, k_2 r) * hx / hy; boundary faces (2 k / r) hy / hx
// and (2 k r) hx / hy.  1 / r and hx / hy come from the host; with
// r = aspect = 1 every factor is an exact 1.
struct AssemblyScale {
  double inv_r, r, aspect, inv_aspect;
  double beta[4];   // west, east, south, north: < 0 Dirichlet, else Robin beta
};

// A boundary face: the Dirichlet coefficient d (wall half a cell away), or
// for a Robin wall (k du/dn + alpha u = 0, beta = alpha times the cell width
// normal to the wall) the series conductance d * beta / (2 k_n + beta);
// beta = 0 is Neumann.
__device__ __forceinline__ double boundary_face(double d, double kn, double beta) {
  return beta < 0.0 ? d : d * (beta / (2.0 * kn + beta));
}

// Writes C, 1/C, W, S of the finest level and a dense copy of k; flags k that
// is not finite and positive.  The tile's coefficients and a halo of one cell
// are read (and their exponential taken) once, into shared memory; each thread
// forms the west and south faces of its cell (each interior face once); the
// east and north faces come from the neighbours through shared memory.  The
// east face of cell q is the same call as the west face of cell q+1, so C is
// what forming all four faces per cell would give.
//
// What bounds it: FP64 instructions, which a warp issues at the same cost
// whatever its active lanes.  The faces beyond the tile and the halo's
// exponentials are therefore dealt to whole warps instead of to every warp's
// last lane, the range check is done on the bits, and with UNIT (r = aspect =
// 1) the multiplications by an exact 1 are left out: 57 -> 38 operations a
// cell (6.5 -> 4.0 ms at 8191^2).
template <typename T, bool UNIT>
__global__ void __launch_bounds__(kAX * kAY) k_assemble(const double* __restrict__ k, int nx,
                                                        int ny, LevelV<T> L,
                                                        double* __restrict__ kcopy, int* derr,
                                                        bool log_k, AssemblyScale f) {
  __shared__ double kt[kAY + 2][kAX + 2];   // k with a halo of one cell
  __shared__ double fw[kAY][kAX + 1];       // west faces, column kAX = east of the tile
  __shared__ double fs[kAY + 1][kAX];       // south faces, row kAY = north of the tile
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int ib = blockIdx.x * kAX, jb = blockIdx.y * kAY;
  const int i0 = ib + tx, j0 = jb + ty;
  const bool in = i0 < nx && j0 < ny;
  const size_t q = size_t(j0) * nx + i0;
  // cell (i, j) of the grid into the tile; warps 0 and 1 add the rows below
  // and above it, warp 2 the columns beside it
  auto cell = [&](int i, int j) {
    if (i >= 0 && i < nx && j >= 0 && j < ny)
      kt[j - jb + 1][i - ib + 1] = cell_k(k, size_t(j) * nx + i, log_k);
  };
  cell(i0, j0);
  if (ty == 0) cell(i0, jb - 1);
  if (ty == 1) cell(i0, jb + kAY);
  if (ty == 2 && tx < 2 * kAY) cell(tx < kAY ? ib - 1 : ib + kAX, jb + tx % kAY);
  __syncthreads();
  auto kx = [&](int x, int y) { return UNIT ? kt[y + 1][x + 1] : kt[y + 1][x + 1] * f.inv_r; };
  auto ky = [&](int x, int y) { return UNIT ? kt[y + 1][x + 1] : kt[y + 1][x + 1] * f.r; };
  // west face of tile cell (x, y), south face likewise; 0 on the boundary and
  // beyond the grid
  auto west = [&](int x, int y) {
    double v = 0.0;
    if (ib + x > 0 && ib + x < nx && jb + y < ny) {
      v = harmonic(kx(x - 1, y), kx(x, y));
      if (!UNIT) v = v * f.aspect;
    }
    fw[y][x] = v;
  };
  auto south = [&](int x, int y) {
    double v = 0.0;
    if (ib + x < nx && jb + y > 0 && jb + y < ny) {
      v = harmonic(ky(x, y - 1), ky(x, y));
      if (!UNIT) v = v * f.inv_aspect;
    }
    fs[y][x] = v;
  };
  west(tx, ty);
  south(tx, ty);
  if (ty == 0 && tx < kAY) west(kAX, tx);
  if (ty == 1) south(tx, kAY);
  __syncthreads();
  if (!in) return;
  const double kc = kt[ty + 1][tx + 1];
  const long long bits = __double_as_longlong(kc);
  if (!(bits > 0 && bits < 0x7FF0000000000000LL)) atomicOr(derr, DEV_BADK);
  kcopy[q] = kc;
  const double aw = fw[ty][tx], as = fs[ty][tx];
  const double ae = fw[ty][tx + 1];
  const double an = fs[ty + 1][tx];
  // boundary faces, in the order west, east, south, north
  double bw = 0.0;
  if (i0 == 0 || i0 == nx - 1 || j0 == 0 || j0 == ny - 1) {
    const double kxc = kx(tx, ty), kyc = ky(tx, ty);
    if (i0 == 0) bw = bw + boundary_face(2.0 * kxc * f.aspect, kxc, f.beta[0]);
    if (i0 == nx - 1) bw = bw + boundary_face(2.0 * kxc * f.aspect, kxc, f.beta[1]);
    if (j0 == 0) bw = bw + boundary_face(2.0 * kyc * f.inv_aspect, kyc, f.beta[2]);
    if (j0 == ny - 1) bw = bw + boundary_face(2.0 * kyc * f.inv_aspect, kyc, f.beta[3]);
  }
  const double c = (((aw + ae) + as) + an) + bw;
  const int o = (j0 + 1) * L.pitch + (i0 + 1);
  L.C[o] = T(c);
  L.iC[o] = T(__drcp_rn(c));
  L.W[o] = T(aw);
  L.S[o] = T(as);
}

// Fine stencil row at plane offset o, as the interpolation formulas use it:
// negated off-diagonals a_X with a_X < 0 (positive matrix entries) lumped into
// the diagonal and a negative row sum sigma dropped,
//   a_X+ = max(a_X, 0),  C_eff = C - sum_X min(a_X, 0) - min(sigma, 0).
// On M-matrix rows with sigma >= 0 (the whole assembled level) this is the
// plain row.  Sums run in the order W, E, S, N, SW, SE, NW, NE.
// Entries below zero are rare (the sign bits tell, in integers), a row sum
// rounded below zero is not.
template <typename T, bool NINE>
struct St {
  T c, w, e, s, n, sw, se, nw, ne;
  __device__ __forceinline__ St(const LevelV<T>& L, int o) {
    const int p = L.pitch;
    c = L.C[o];
    w = L.W[o];
    e = L.W[o + 1];
    s = L.S[o];
    n = L.S[o + p];
    if (NINE) {
      sw = L.SW[o];
      ne = L.SW[o + 1 + p];
      nw = L.NW[o];
      se = L.NW[o + 1 - p];
    } else {
      sw = se = nw = ne = T(0);
    }
    T total = ((w + e) + s) + n;
    if (NINE) total = (((total + sw) + se) + nw) + ne;
    const T sigma = c - total;
    bool lump = sign_bit(w) || sign_bit(e) || sign_bit(s) || sign_bit(n);
    if (NINE) lump = lump || sign_bit(sw) || sign_bit(se) || sign_bit(nw) || sign_bit(ne);
    if (lump) {
      St t = *this;
      t.drop_negative();
      *this = t;
    }
    c = c - (below_zero(sigma) ? sigma : T(0));
  }
  __device__ __noinline__ void drop_negative() {
    const T z = T(0);
    const T neg = ((((((((z + fmin(w, z)) + fmin(e, z)) + fmin(s, z)) + fmin(n, z)) + fmin(sw, z)) +
                     fmin(se, z)) + fmin(nw, z)) + fmin(ne, z));
    c = c - neg;
    w = fmax(w, z);
    e = fmax(e, z);
    s = fmax(s, z);
    n = fmax(n, z);
    sw = fmax(sw, z);
    se = fmax(se, z);
    nw = fmax(nw, z);
    ne = fmax(ne, z);
  }
};

// x-edge point: collapse the fine row in y (flux balance along x).
template <typename T, bool NINE>
__device__ __forceinline__ void xedge(const LevelV<T>& L, int o, T& ww, T& we, int* derr,
                                      int lbit) {
  St<T, NINE> a(L, o);
  const T den = (a.c - a.s) - a.n;
  if (!(den > T(0))) atomicOr(derr, DEV_BADDEN | lbit);
  const auto d = denominator(den);
  ww = divide(NINE ? (a.w + a.sw) + a.nw : a.w, d);
  we = divide(NINE ? (a.e + a.se) + a.ne : a.e, d);
}

// y-edge point: collapse the fine row in x.
template <typename T, bool NINE>
__device__ __forceinline__ void yedge(const LevelV<T>& L, int o, T& ws, T& wn, int* derr,
                                      int lbit) {
  St<T, NINE> a(L, o);
  const T den = (a.c - a.w) - a.e;
  if (!(den > T(0))) atomicOr(derr, DEV_BADDEN | lbit);
  const auto d = denominator(den);
  ws = divide(NINE ? (a.s + a.sw) + a.se : a.s, d);
  wn = divide(NINE ? (a.n + a.nw) + a.ne : a.n, d);
}

// One thread per coarse-grid index (I, J), 0 <= I <= ncx, 0 <= J <= ncy
// (ncx = floor(nx / 2)).  Computes the weights of the x-edge point
// (2I+1, 2J), the y-edge point (2I, 2J+1) and the centre point (2I+1, 2J+1)
// where those fine points exist: on an even side the last fine point is a
// coarse point, so column 2I+1 (or row 2J+1) may lie beyond the grid; its
// weights stay zero and nothing is read there.  The centre point's other two
// edge neighbours, (2I+1, 2J+2) and (2I+2, 2J+1), come from the neighbouring
// threads through shared memory; a whole warp each computes those beyond the
// tile.
//
// What bounds it: FP64 instructions (small levels: the chain of divisions).
// Each edge once instead of twice, one reciprocal per denominator instead of a
// division per weight, comparisons in integers: 210 -> 75 operations per
// coarse point of a 5-point level, 350 -> 100 of a 9-point one
// (9088 x 568: 548 -> 172 us and, for all coarser levels, 355 -> 127 us).
template <typename T, bool NINE>
__global__ void __launch_bounds__(kAX * kAY) k_interp_weights(LevelV<T> F, int ncx, int ncy,
                                                              int* derr, int level) {
  __shared__ T xw[kAY + 1][kAX], xe[kAY + 1][kAX];   // x-edges (2I+1, 2J)
  __shared__ T ys[kAY][kAX + 1], yn[kAY][kAX + 1];   // y-edges (2I, 2J+1)
  const int lbit = 1 << (8 + level);
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int Ib = blockIdx.x * kAX, Jb = blockIdx.y * kAY;
  const int I = Ib + tx, J = Jb + ty;
  const int p = F.pitch, cp = F.cpitch;
  auto x_at = [&](int x, int y) {
    const int i = 2 * (Ib + x) + 1, j = 2 * (Jb + y);
    T w = T(0), e = T(0);
    if (i <= F.nx && j >= 2 && j <= 2 * ncy) xedge<T, NINE>(F, j * p + i, w, e, derr, lbit);
    xw[y][x] = w;
    xe[y][x] = e;
  };
  auto y_at = [&](int x, int y) {
    const int i = 2 * (Ib + x), j = 2 * (Jb + y) + 1;
    T s = T(0), n = T(0);
    if (j <= F.ny && i >= 2 && i <= 2 * ncx) yedge<T, NINE>(F, j * p + i, s, n, derr, lbit);
    ys[y][x] = s;
    yn[y][x] = n;
  };
  x_at(tx, ty);
  y_at(tx, ty);
  if (ty == 0) x_at(tx, kAY);
  if (ty == 1 && tx < kAY) y_at(kAX, tx);
  __syncthreads();
  if (I > ncx || J > ncy) return;
  const int c = J * cp + I;
  const bool col_odd = 2 * I + 1 <= F.nx;   // fine column 2I+1 exists
  const bool row_odd = 2 * J + 1 <= F.ny;   // fine row 2J+1 exists
  if (col_odd && J >= 1) {
    F.P[XW][c] = xw[ty][tx];
    F.P[XE][c] = xe[ty][tx];
  }
  if (row_odd && I >= 1) {
    F.P[YS][c] = ys[ty][tx];
    F.P[YN][c] = yn[ty][tx];
  }
  if (!(col_odd && row_odd)) return;
  // centre (2I+1, 2J+1): the fine equation with the edge neighbours replaced
  // by their interpolants.
  St<T, NINE> a(F, (2 * J + 1) * p + 2 * I + 1);
  const auto d = denominator(a.c);
  F.P[CSW][c] = divide((a.sw + a.w * ys[ty][tx]) + a.s * xw[ty][tx], d);
  F.P[CSE][c] = divide((a.se + a.e * ys[ty][tx + 1]) + a.s * xe[ty][tx], d);
  F.P[CNW][c] = divide((a.nw + a.w * yn[ty][tx]) + a.n * xw[ty + 1][tx], d);
  F.P[CNE][c] = divide((a.ne + a.e * yn[ty][tx + 1]) + a.n * xe[ty + 1][tx], d);
}

// Matrix entry A[p, p + (dx, dy)] of the fine operator at plane offset o.
template <typename T, bool NINE>
__device__ __forceinline__ T aentry(const LevelV<T>& L, int o, int dx, int dy) {
  const int p = L.pitch;
  if (dx == 0 && dy == 0) return L.C[o];
  if (dy == 0) return dx < 0 ? -L.W[o] : -L.W[o + 1];
  if (dx == 0) return dy < 0 ? -L.S[o] : -L.S[o + p];
  if (!NINE) return T(0);
  if (dx < 0 && dy < 0) return -L.SW[o];
  if (dx > 0 && dy > 0) return -L.SW[o + 1 + p];
  if (dx < 0 && dy > 0) return -L.NW[o];
  return -L.NW[o + 1 - p];
}

// Galerkin entry A_c[(I,J), (I+DX, J+DY)] = sum_{p near 2I} P(p, I)
// sum_{q near p} A(p, q) P(q, I + D).  Terms whose q lies outside the support
// of P(., I + D) are removed at compile time after unrolling.
template <typename T, bool NINE, int DX, int DY>
__device__ __forceinline__ T rap_entry(const LevelV<T>& F, int I, int J) {
  const int p = F.pitch, cp = F.cpitch;
  const int c = J * cp + I;
  const int ct = (J + DY) * cp + (I + DX);
  T sum = T(0);
#pragma unroll
  for (int py = -1; py <= 1; ++py) {
#pragma unroll
    for (int px = -1; px <= 1; ++px) {
      // fine points beyond an even side do not exist (their weights are 0)
      if (2 * I + px > F.nx || 2 * J + py > F.ny) continue;
      const int o = (2 * J + py) * p + (2 * I + px);
      T inner = T(0);
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy) {
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
          const int rx = px + dx - 2 * DX, ry = py + dy - 2 * DY;
          if (rx < -1 || rx > 1 || ry < -1 || ry > 1) continue;
          if (!NINE && dx != 0 && dy != 0) continue;
          inner = fma(aentry<T, NINE>(F, o, dx, dy), pweight<T>(F.P, cp, rx, ry, ct), inner);
        }
      }
      sum = fma(pweight<T>(F.P, cp, px, py, c), inner, sum);
    }
  }
  return sum;
}

// One thread per interior coarse point: the five stored planes of A_{l-1}.
template <typename T, bool NINE>
__global__ void k_rap(LevelV<T> F, LevelV<T> Cc) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x + 1;
  const int J = blockIdx.y + 1;
  if (I > Cc.nx) return;
  const int o = J * Cc.pitch + I;
  const T cc = rap_entry<T, NINE, 0, 0>(F, I, J);
  Cc.C[o] = cc;
  Cc.iC[o] = T(1) / cc;
  Cc.W[o] = I > 1 ? -rap_entry<T, NINE, -1, 0>(F, I, J) : T(0);
  Cc.S[o] = J > 1 ? -rap_entry<T, NINE, 0, -1>(F, I, J) : T(0);
  Cc.SW[o] = (I > 1 && J > 1) ? -rap_entry<T, NINE, -1, -1>(F, I, J) : T(0);
  Cc.NW[o] = (I > 1 && J < Cc.ny) ? -rap_entry<T, NINE, -1, 1>(F, I, J) : T(0);
}

// Dense A_0 (FP64) from the coarsest planes, then an in-place right-looking
// Cholesky factorisation in one thread block; stores 1/L[i][i] and the
// diagonal of A_0 too.  The
// matrix is worked on in shared memory where it fits (SMEM, up to 160
// unknowns: rows of n | 1, free of bank conflicts), else in `a`.
//
// What bounds it: the chain of n square roots and reciprocals and one SM's
// FP64 rate in the updates.  Threads are 16 x 32 over the trailing matrix, no
// index divisions: 70 unknowns 121 -> 90 us.
constexpr size_t kDenseSmem = 160 * 161 * sizeof(double);

inline size_t dense_smem(int n) {
  const size_t bytes = size_t(n) * (n | 1) * sizeof(double);
  return bytes <= kDenseSmem ? bytes : 0;
}

template <typename T, bool SMEM>
__global__ void __launch_bounds__(512) k_coarse_factor(LevelV<T> L0, double* __restrict__ a,
                                                       double* __restrict__ idiag, int* derr) {
  extern __shared__ double dense[];
  const int nx = L0.nx, ny = L0.ny, n = nx * ny, p = L0.pitch;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, rows = blockDim.x >> 5;
  double* const m = SMEM ? dense : a;
  const int mp = SMEM ? n | 1 : n;
  for (int i = ty; i < n; i += rows)
    for (int j = tx; j < n; j += 32) m[size_t(i) * mp + j] = 0.0;
  __syncthreads();
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    const int i = r % nx + 1, j = r / nx + 1, o = j * p + i;
    m[size_t(r) * mp + r] = double(L0.C[o]);
    idiag[n + r] = double(L0.C[o]);
    auto put = [&](int di, int dj, double v) {
      const int ii = i + di, jj = j + dj;
      if (ii < 1 || ii > nx || jj < 1 || jj > ny) return;
      m[size_t(r) * mp + (jj - 1) * nx + (ii - 1)] = -v;
    };
    put(-1, 0, double(L0.W[o]));
    put(1, 0, double(L0.W[o + 1]));
    put(0, -1, double(L0.S[o]));
    put(0, 1, double(L0.S[o + p]));
    if (L0.SW) {
      put(-1, -1, double(L0.SW[o]));
      put(1, 1, double(L0.SW[o + 1 + p]));
      put(-1, 1, double(L0.NW[o]));
      put(1, -1, double(L0.NW[o + 1 - p]));
    }
  }
  __syncthreads();
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    if (threadIdx.x == 0) {
      const double d = m[size_t(k) * mp + k];
      if (!(d > 0.0)) {
        bad = 1;
        atomicOr(derr, DEV_NOTSPD);
      }
      const double s = sqrt(d > 0.0 ? d : 1.0);
      m[size_t(k) * mp + k] = s;
      idiag[k] = 1.0 / s;
    }
    __syncthreads();
    if (bad) return;
    const double inv = idiag[k];
    for (int i = k + 1 + threadIdx.x; i < n; i += blockDim.x) m[size_t(i) * mp + k] *= inv;
    __syncthreads();
    for (int i = k + 1 + ty; i < n; i += rows)
      for (int j = k + 1 + tx; j <= i; j += 32)
        m[size_t(i) * mp + j] -= m[size_t(i) * mp + k] * m[size_t(j) * mp + k];
    __syncthreads();
  }
  for (int i = ty; i < n; i += rows)
    for (int j = tx; j < n; j += 32) a[size_t(i) * n + j] = j > i ? 0.0 : m[size_t(i) * mp + j];
}

// The inverse of the coarsest operator from its factor, and its measure (see
// CoarseSolve; zeroed by the caller), one column per
// block: forward and backward substitution of a unit vector, one barrier per
// column of the factor.  A product with it takes the place of a substitution
// in every V-cycle: the substitution's 2 n dependent steps of two FP64
// operations each (9 unknowns: 3.5 us of a 25 us sub-cycle; 70 unknowns: 20
// us) become one short chain per unknown.  The factor is read into shared
// memory where it fits: a step's column then costs no trip to L2 (70
// unknowns: 43 -> 31 us).
template <bool SMEM>
__global__ void __launch_bounds__(128) k_coarse_inverse(const double* __restrict__ lo,
                                                        const double* __restrict__ idiag, int n,
                                                        double* __restrict__ inv,
                                                        double* __restrict__ measure) {
  extern __shared__ double dense[];
  const int c = blockIdx.x;
  const int mp = SMEM ? n | 1 : n;
  double* const v = dense + (SMEM ? n * mp : 0);
  double* const y = v + n;
  double* const id = y + n;
  if (SMEM)
    for (int i = threadIdx.x >> 5; i < n; i += 4)
      for (int j = threadIdx.x & 31; j <= i; j += 32) dense[i * mp + j] = lo[size_t(i) * n + j];
  const double* const m = SMEM ? dense : lo;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    v[i] = i == c ? 1.0 : 0.0;
    y[i] = 0.0;
    id[i] = idiag[i];
  }
  for (int j = c; j < n; ++j) {
    __syncthreads();
    const double yj = v[j] * id[j];
    if (threadIdx.x == 0) y[j] = yj;
    for (int i = j + 1 + threadIdx.x; i < n; i += blockDim.x)
      v[i] = fma(-m[size_t(i) * mp + j], yj, v[i]);
  }
  for (int j = n - 1; j >= 0; --j) {
    __syncthreads();
    const double xj = y[j] * id[j];
    if (threadIdx.x == 0) {
      inv[size_t(c) * n + j] = xj;
      if (j == c) raise(measure, xj * idiag[n + c]);
    }
    for (int i = threadIdx.x; i < j; i += blockDim.x) y[i] = fma(-m[size_t(j) * mp + i], xj, y[i]);
  }
}

template <typename T>
int coarse_factor(Hierarchy* h, const LevelV<T>& l0, cudaStream_t s) {
  int* derr = &h->sc->err;
  const size_t smem = dense_smem(h->n0), vectors = 3 * h->n0 * sizeof(double);
  if (smem) {
    if (!use_shared(k_coarse_factor<T, true>, smem) || !use_shared(k_coarse_inverse<true>, smem + vectors))
      return BMG_ECUDA;
    k_coarse_factor<T, true><<<1, 512, smem, s>>>(l0, h->chol, h->chol_idiag, derr);
    k_coarse_inverse<true><<<h->n0, 128, smem + vectors, s>>>(h->chol, h->chol_idiag, h->n0, h->cinv, &h->sc->measure);
  } else {
    k_coarse_factor<T, false><<<1, 512, 0, s>>>(l0, h->chol, h->chol_idiag, derr);
    k_coarse_inverse<false><<<h->n0, 128, vectors, s>>>(h->chol, h->chol_idiag, h->n0, h->cinv, &h->sc->measure);
  }
  count_launch(2);
  return cudaGetLastError() == cudaSuccess ? 0 : BMG_ECUDA;
}

__global__ void k_downcast(LevelV<double> D, LevelV<float> F) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x + 1;
  const int j = blockIdx.y + 1;
  if (i > D.nx) return;
  const int od = j * D.pitch + i, of = j * F.pitch + i;
  F.C[of] = float(D.C[od]);
  F.iC[of] = float(D.iC[od]);
  F.W[of] = float(D.W[od]);
  F.S[of] = float(D.S[od]);
}

template <typename T>
__global__ void k_pack(const double* __restrict__ src, T* __restrict__ dst, int nx, int pitch) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (i >= nx) return;
  dst[(j + 1) * pitch + i + 1] = T(src[size_t(j) * nx + i]);
}

template <typename T>
__global__ void k_unpack(const T* __restrict__ src, double* __restrict__ dst, int nx, int pitch) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (i >= nx) return;
  dst[size_t(j) * nx + i] = double(src[(j + 1) * pitch + i + 1]);
}

// Backward of the assembly, one thread per cell (dense arrays):
// g_c = -k_c [ sum_faces 2 k_n^2/(k_c + k_n)^2 (u_c - u_n)(lam_c - lam_n)
//              + (#boundary faces) 2 u_c lam_c ].
__global__ void k_assemble_backward(const double* __restrict__ k, const double* __restrict__ u,
                                    const double* __restrict__ lam, double* __restrict__ g,
                                    int nx, int ny) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (i >= nx) return;
  const size_t q = size_t(j) * nx + i;
  const double kc = k[q], uc = u[q], lc = lam[q];
  double acc = 0.0;
  int nb = 0;
  auto face = [&](size_t qn) {
    const double kn = k[qn];
    const double s = kc + kn;
    acc += 2.0 * kn * kn / (s * s) * ((uc - u[qn]) * (lc - lam[qn]));
  };
  if (i > 0) face(q - 1); else ++nb;
  if (i < nx - 1) face(q + 1); else ++nb;
  if (j > 0) face(q - nx); else ++nb;
  if (j < ny - 1) face(q + nx); else ++nb;
  acc += double(nb) * 2.0 * uc * lc;
  g[q] = -kc * acc;
}

}  // namespace

template <typename T>
int launch_assemble(const double* k, int nx, int ny, LevelV<T> L, double* kcopy, int* derr,
                    bool log_k, double r, double aspect, const double* bc_beta, cudaStream_t s) {
  const AssemblyScale f{1.0 / r, r, aspect, 1.0 / aspect,
                        {bc_beta[0], bc_beta[1], bc_beta[2], bc_beta[3]}};
  const dim3 grid(cdiv(nx, kAX), cdiv(ny, kAY)), block(kAX, kAY);
  if (r == 1.0 && aspect == 1.0)
    k_assemble<T, true><<<grid, block, 0, s>>>(k, nx, ny, L, kcopy, derr, log_k, f);
  else
    k_assemble<T, false><<<grid, block, 0, s>>>(k, nx, ny, L, kcopy, derr, log_k, f);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : BMG_ECUDA;
}

template <typename T>
int launch_interp_weights(const LevelV<T>& fine, bool nine, int* derr, int level, cudaStream_t s) {
  const int ncx = fine.nx / 2, ncy = fine.ny / 2;
  const dim3 grid(cdiv(ncx + 1, kAX), cdiv(ncy + 1, kAY)), block(kAX, kAY);
  if (nine)
    k_interp_weights<T, true><<<grid, block, 0, s>>>(fine, ncx, ncy, derr, level);
  else
    k_interp_weights<T, false><<<grid, block, 0, s>>>(fine, ncx, ncy, derr, level);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : BMG_ECUDA;
}

template <typename T>
int launch_rap(const LevelV<T>& fine, bool nine, LevelV<T> coarse, cudaStream_t s) {
  dim3 grid(cdiv(coarse.nx, 128), coarse.ny);
  if (nine)
    k_rap<T, true><<<grid, 128, 0, s>>>(fine, coarse);
  else
    k_rap<T, false><<<grid, 128, 0, s>>>(fine, coarse);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : BMG_ECUDA;
}

int launch_coarse_factor(Hierarchy* h, const LevelV<double>* l0d, const LevelV<float>* l0f,
                         cudaStream_t s) {
  return l0d ? coarse_factor(h, *l0d, s) : coarse_factor(h, *l0f, s);
}

int launch_downcast_fine(const LevelV<double>& d, LevelV<float> f, cudaStream_t s) {
  k_downcast<<<dim3(cdiv(d.nx, kTB), d.ny), kTB, 0, s>>>(d, f);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? 0 : BMG_ECUDA;
}

template <typename T>
void launch_pack(const double* src, T* dst, int nx, int ny, int pitch, cudaStream_t s) {
  k_pack<T><<<dim3(cdiv(nx, kTB), ny), kTB, 0, s>>>(src, dst, nx, pitch);
  count_launch();
}

template <typename T>
void launch_unpack(const T* src, double* dst, int nx, int ny, int pitch, cudaStream_t s) {
  k_unpack<T><<<dim3(cdiv(nx, kTB), ny), kTB, 0, s>>>(src, dst, nx, pitch);
  count_launch();
}

void launch_assemble_backward(const double* k, const double* u, const double* lam, double* g,
                              int nx, int ny, cudaStream_t s) {
  k_assemble_backward<<<dim3(cdiv(nx, kTB), ny), kTB, 0, s>>>(k, u, lam, g, nx, ny);
  count_launch();
}

template int launch_assemble<double>(const double*, int, int, LevelV<double>, double*, int*,
                                     bool, double, double, const double*, cudaStream_t);
template int launch_interp_weights<double>(const LevelV<double>&, bool, int*, int, cudaStream_t);
template int launch_interp_weights<float>(const LevelV<float>&, bool, int*, int, cudaStream_t);
template int launch_rap<double>(const LevelV<double>&, bool, LevelV<double>, cudaStream_t);
template int launch_rap<float>(const LevelV<float>&, bool, LevelV<float>, cudaStream_t);
template void launch_pack<double>(const double*, double*, int, int, int, cudaStream_t);
template void launch_pack<float>(const double*, float*, int, int, int, cudaStream_t);
template void launch_unpack<double>(const double*, double*, int, int, int, cudaStream_t);
template void launch_unpack<float>(const float*, double*, int, int, int, cudaStream_t);

}  // namespace bmg
