// Vector work of the preconditioned conjugate gradients on the finest level,
// shared by the single-problem and the batched solver, and the conversions
// between FP32 and FP64 it needs.
//
// What bounds it.  GB300 runs about 600 G FP64 instructions a second, and a
// conversion between float and double takes an FP64 slot too (measured: 594 G
// a second, as a fused multiply-add), so of an iteration's passes A p (six
// FP64 operations a point) is bound by that pipe and the others by a mix of
// pipe and memory.  Hence the conversions below, which take integer
// instructions instead (same results), and no pass of their own for
// z = M^{-1} r with an FP32 preconditioner: the passes that use z form it
// from the FP32 iterate.
//
// A pass deals the level's pairs of points (i, i + 1), i odd, to the blocks
// in runs of kKT, a pair per thread: interior rows start on 128-byte
// boundaries, so a pair is one 16-byte access, and no block idles on a short
// or a last row (rows dealt whole left a quarter of 608 blocks idle on 1023
// rows).  The order is fixed, so the sums are deterministic.
#pragma once

#include "bmg_internal.h"

namespace bmg {

constexpr int kKT = 256;   // threads of a pass

// The conversions of the rare values, out of line: the compiler would
// otherwise execute the conversion for every value and select afterwards.
static __device__ __noinline__ float to_float_rare(double d) { return float(d); }
static __device__ __noinline__ double to_double_rare(float f) { return double(f); }

// float(d), round to nearest even.  Normal results take the integer path: the
// float's exponent and upper mantissa bits are a funnel shift of the
// double's words, rebiased, plus one where the 29 bits below round up (a
// carry runs into the exponent as it should).
__device__ __forceinline__ float to_float(double d) {
  const unsigned hi = unsigned(__double2hiint(d)), lo = unsigned(__double2loint(d));
  const unsigned e = (hi >> 20) & 0x7FFu;
  if (e - 897u >= 254u && (hi << 1 | lo) != 0u) return to_float_rare(d);   // subnormal, overflow, infinity, NaN
  unsigned u = (__funnelshift_l(lo, hi, 3) - (896u << 23)) & 0x7FFFFFFFu;
  u += (lo << 3) + (u & 1u) > 0x80000000u ? 1u : 0u;
  if ((hi << 1 | lo) == 0u) u = 0u;
  return __uint_as_float(u | (hi & 0x80000000u));
}

// double(f) (exact); zeros and normal numbers take the integer path.
__device__ __forceinline__ double to_double(float f) {
  const unsigned u = __float_as_uint(f), m = u & 0x7FFFFFFFu;
  if (m - 0x00800000u >= 0x7F000000u && m != 0u) return to_double_rare(f);   // subnormal, infinity, NaN
  const unsigned hi = m ? (m >> 3) + (896u << 20) : 0u;
  return __hiloint2double(int(hi | (u & 0x80000000u)), int(u << 29));
}

__device__ __forceinline__ double krylov_block_sum(double v) {
  __shared__ double red[kKT / 32];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) red[w] = v;
  __syncthreads();
  v = lane < kKT / 32 ? red[lane] : 0.0;
  if (w == 0) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  }
  return v;
}

// Calls f(j, i, two) for the pairs of block `b` of `nb` (two: i + 1 is in the
// grid).
__host__ __device__ __forceinline__ int pair_runs(int nx, int ny) {
  return int((size_t((nx + 1) / 2) * ny + kKT - 1) / kKT);
}
template <class F>
__device__ __forceinline__ void for_pairs(int nx, int ny, int b, int nb, F f) {
  const unsigned per = unsigned(nx + 1) / 2, n = per * unsigned(ny);
  for (unsigned t = unsigned(b) * kKT + threadIdx.x; t < n; t += unsigned(nb) * kKT) {
    const unsigned jj = t / per;
    const int i = 2 * int(t - jj * per) + 1;
    f(int(jj) + 1, i, i + 1 <= nx);
  }
}

// The same with the loads of a thread's next pair in flight while it works on
// one: load(j, i) fetches a pair's values, work(j, i, two, values) uses them.
template <class L, class W>
__device__ __forceinline__ void for_pairs_ahead(int nx, int ny, int b, int nb, L load, W work) {
  const unsigned per = unsigned(nx + 1) / 2, n = per * unsigned(ny), step = unsigned(nb) * kKT;
  unsigned t = unsigned(b) * kKT + threadIdx.x;
  if (t >= n) return;
  int j = int(t / per) + 1, i = 2 * int(t % per) + 1;
  auto v = load(j, i);
  for (;;) {
    const unsigned tn = t + step;
    const bool more = tn < n;
    auto vn = v;
    int jn = j, in = i;
    if (more) {
      jn = int(tn / per) + 1;
      in = 2 * int(tn % per) + 1;
      vn = load(jn, in);
    }
    work(j, i, i + 1 <= nx, v);
    if (!more) return;
    v = vn;
    j = jn;
    i = in;
    t = tn;
  }
}

__device__ __forceinline__ double2 load2(const double* p) { return *reinterpret_cast<const double2*>(p); }
__device__ __forceinline__ void store2(double* p, double a, double b, bool two) {
  if (two)
    *reinterpret_cast<double2*>(p) = make_double2(a, b);
  else
    *p = a;
}

// What resid_value (5-point) reads for the pair at o, and its two values.
struct ResidPair {
  double2 c, w, s, n, xc, xs, xn;
  double w2, xw, xe;
};
__device__ __forceinline__ ResidPair load_resid(const LevelV<double>& L, const double* x, int o) {
  const int p = L.pitch;
  return ResidPair{load2(L.C + o),     load2(L.W + o),     load2(L.S + o), load2(L.S + o + p), load2(x + o),
                   load2(x + o - p), load2(x + o + p), L.W[o + 2],     x[o - 1],           x[o + 2]};
}
__device__ __forceinline__ double2 resid_pair(const ResidPair& v, double2 b) {
  double2 r;
  r.x = fma(-v.c.x, v.xc.x, b.x);
  r.y = fma(-v.c.y, v.xc.y, b.y);
  r.x = fma(v.w.x, v.xw, r.x);
  r.y = fma(v.w.y, v.xc.x, r.y);
  r.x = fma(v.w.y, v.xc.y, r.x);
  r.y = fma(v.w2, v.xe, r.y);
  r.x = fma(v.s.x, v.xs.x, r.x);
  r.y = fma(v.s.y, v.xs.y, r.y);
  r.x = fma(v.n.x, v.xn.x, r.x);
  r.y = fma(v.n.y, v.xn.y, r.y);
  return r;
}

// A x of the pair: the terms of resid_value for b = 0 with their signs turned
// (so the same values, and no operation to negate them).
__device__ __forceinline__ double2 apply_pair(const ResidPair& v) {
  double2 r;
  r.x = v.c.x * v.xc.x;
  r.y = v.c.y * v.xc.y;
  r.x = fma(-v.w.x, v.xw, r.x);
  r.y = fma(-v.w.y, v.xc.x, r.y);
  r.x = fma(-v.w.y, v.xc.y, r.x);
  r.y = fma(-v.w2, v.xe, r.y);
  r.x = fma(-v.s.x, v.xs.x, r.x);
  r.y = fma(-v.s.y, v.xs.y, r.y);
  r.x = fma(-v.n.x, v.xn.x, r.x);
  r.y = fma(-v.n.y, v.xn.y, r.y);
  return r;
}

struct PcgVec {
  double *x, *b, *p, *q;   // iterate, right-hand side, direction, A p
};

// One pass over the pairs of block b of nb; the block's partial sum.  The
// finest level's b plane holds r; z is its x plane, or (F: the FP32 finest
// level) ||r|| times the FP32 iterate e.
//  INIT r = b - A x;            r.r     AP  q = A p;        p.q
//  XR   x += alpha p, r -= alpha q; r.r     RZ  r.z (F: r.e)     P   p = z + beta p
// A prescaled level also gets b/C; zero_z: z = 0 (cycles that read it).
enum { K_INIT = 0, K_AP, K_XR, K_RZ, K_P };

template <int WHAT, bool F32>
__device__ __forceinline__ double krylov_pass(const LevelV<double>& L, const LevelV<float>* F, const PcgVec& v,
                                              const Scalars* sc, bool zero_z, int b, int nb) {
  const int pitch = L.pitch;
  double acc = 0.0;
  double* const rp = L.b;
  if constexpr (WHAT == K_INIT || WHAT == K_XR) {
    double *const pre = L.PR[PR_B], *const zp = L.x;
    const double* const icp = L.iC;
    auto set_r = [&](int o, double r0, double r1, bool two) {
      store2(rp + o, r0, r1, two);
      if (pre) {
        const double2 ic = load2(icp + o);
        store2(pre + o, r0 * ic.x, r1 * ic.y, two);
      }
      if (zero_z) store2(zp + o, 0.0, 0.0, two);
      acc = fma(r0, r0, acc);
      if (two) acc = fma(r1, r1, acc);
    };
    if constexpr (WHAT == K_INIT) {
      for_pairs(L.nx, L.ny, b, nb, [&](int j, int i, bool two) {
        const int o = j * pitch + i;
        const double2 r = resid_pair(load_resid(L, v.x, o), load2(v.b + o));
        set_r(o, r.x, r.y, two);
      });
    } else {
      const double alpha = sc->alpha;
      struct V {
        double2 p, x, q, r;
      };
      for_pairs_ahead(
          L.nx, L.ny, b, nb,
          [&](int j, int i) {
            const int o = j * pitch + i;
            return V{load2(v.p + o), load2(v.x + o), load2(v.q + o), load2(rp + o)};
          },
          [&](int j, int i, bool two, const V& a) {
            const int o = j * pitch + i;
            store2(v.x + o, fma(alpha, a.p.x, a.x.x), fma(alpha, a.p.y, a.x.y), two);
            set_r(o, fma(-alpha, a.q.x, a.r.x), fma(-alpha, a.q.y, a.r.y), two);
          });
    }
  } else if constexpr (WHAT == K_AP) {
    for_pairs_ahead(
        L.nx, L.ny, b, nb, [&](int j, int i) { return load_resid(L, v.p, j * pitch + i); },
        [&](int j, int i, bool two, const ResidPair& a) {
          const double2 q = apply_pair(a);
          store2(v.q + j * pitch + i, q.x, q.y, two);
          acc = fma(a.xc.x, q.x, acc);
          if (two) acc = fma(a.xc.y, q.y, acc);
        });
  } else {
    const float* const fx = F32 ? F->x : nullptr;
    const int fpitch = F32 ? F->pitch : 0;
    const double* const other = WHAT == K_RZ ? rp : v.p;
    const double scale = WHAT == K_P && F32 ? sc->rnorm : 1.0, beta = WHAT == K_P ? sc->beta : 0.0;
    struct V {
      double2 a, z;
      float2 e;
    };
    for_pairs_ahead(
        L.nx, L.ny, b, nb,
        [&](int j, int i) {
          const int o = j * pitch + i;
          V q;
          q.a = load2(other + o);
          if (F32)
            q.e = *reinterpret_cast<const float2*>(fx + j * fpitch + i);
          else
            q.z = load2(L.x + o);
          return q;
        },
        [&](int j, int i, bool two, const V& q) {
          const double e0 = F32 ? to_double(q.e.x) : q.z.x, e1 = F32 ? to_double(q.e.y) : q.z.y;
          if (WHAT == K_RZ) {
            acc = fma(q.a.x, e0, acc);
            if (two) acc = fma(q.a.y, e1, acc);
          } else {
            const double z0 = F32 ? scale * e0 : e0, z1 = F32 ? scale * e1 : e1;
            store2(v.p + j * pitch + i, fma(beta, q.a.x, z0), fma(beta, q.a.y, z1), two);
          }
        });
  }
  return acc;
}

// The FP32 preconditioner's right-hand side r / ||r|| (zero_x: and a zero
// iterate, for cycles that read it).
__device__ __forceinline__ void krylov_cast(const LevelV<double>& L, const LevelV<float>& F, const Scalars* sc,
                                            bool zero_x, int b, int nb) {
  const double inv = sc->inv;
  const int pitch = L.pitch, fpitch = F.pitch;
  const double* const rp = L.b;
  float *const fb = F.b, *const fx = F.x;
  for_pairs_ahead(
      L.nx, L.ny, b, nb, [&](int j, int i) { return load2(rp + j * pitch + i); },
      [&](int j, int i, bool two, const double2& r) {
        const int of = j * fpitch + i;
        const float f0 = to_float(r.x * inv), f1 = to_float(r.y * inv);
        if (two) {
          *reinterpret_cast<float2*>(fb + of) = make_float2(f0, f1);
          if (zero_x) *reinterpret_cast<float2*>(fx + of) = make_float2(0.0f, 0.0f);
        } else {
          fb[of] = f0;
          if (zero_x) fx[of] = 0.0f;
        }
      });
}

}  // namespace bmg
