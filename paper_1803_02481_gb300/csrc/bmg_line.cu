// Zebra line Gauss-Seidel on full grids (the per-line arithmetic is in
// bmg_line.cuh): setup-time factorisation of every line, and one sweep as
// four launches per (direction, colour) step -- right-hand sides, block
// solves, separator chains, final update.
#include <type_traits>

#include "bmg_line.cuh"

namespace bmg {

namespace {

__host__ __device__ inline int cdiv(long a, long b) { return int((a + b - 1) / b); }

constexpr int kPT = 256;        // threads of the point-parallel kernels
constexpr int kBT = 128;        // threads of the block-parallel kernels

// Point-parallel index space of one colour: the fast grid axis runs along
// the contiguous direction of the plane (the points of a row for x-lines,
// the lines of the colour for y-lines).  Calls f(q, k) for every point.
template <int DIR, class F>
__device__ __forceinline__ void for_colour_points(const LineGeo& g, int colour, F f) {
  const int nlc = line_count(g.nl, colour);
  const int fast = DIR == 0 ? g.n : nlc, slow = DIR == 0 ? nlc : g.n;
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= fast) return;
  for (int b = blockIdx.y; b < slow; b += gridDim.y) {
    const int li = DIR == 0 ? b : a, k = (DIR == 0 ? a : b) + 1;
    f(2 * li + colour + 1, k);
  }
}

template <typename T, int DIR, bool NINE>
__global__ void __launch_bounds__(kPT) k_line_rhs(LevelV<T> L, int colour,
                                                  const T* __restrict__ xs) {
  griddep_wait();
  const LineGeo g = line_geo<DIR>(L);
  T* G = line_scratch<DIR>(L);
  for_colour_points<DIR>(g, colour, [&](int q, int k) {
    G[line_fbase<DIR>(L, q) + k * g.fes] = line_rhs<T, DIR, NINE>(L, xs, q * g.ls + k * g.es);
  });
}

// Block-parallel: the fast axis runs over blocks of a row (x-lines) or over
// the lines of the colour (y-lines).
template <typename T, int DIR>
__global__ void __launch_bounds__(kBT) k_line_blocks(LevelV<T> L, int colour) {
  griddep_wait();
  const LineGeo g = line_geo<DIR>(L);
  const int nlc = line_count(g.nl, colour), nb = g.n / kLineM + 1;
  const int fast = DIR == 0 ? nb : nlc, slow = DIR == 0 ? nlc : nb;
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= fast) return;
  for (int b = blockIdx.y; b < slow; b += gridDim.y) {
    const int li = DIR == 0 ? b : a, bb = DIR == 0 ? a : b;
    line_block_solve<T, DIR>(L, 2 * li + colour + 1, bb);
  }
}

// x-lines: one thread block per segment of kXSeg blocks of a row.  The
// segment's right-hand sides and factors are loaded with contiguous accesses
// into shared memory (one word of padding per block of kLineM points, so the
// threads' block-strided reads hit distinct banks), each thread substitutes
// its block there, and the solutions go back with contiguous stores.
constexpr int kXSeg = 128;
constexpr int kXPts = kXSeg * kLineM;
constexpr int kXPad = kXSeg * (kLineM + 1);

template <typename T>
size_t xblocks_smem() { return 4 * size_t(kXPad) * sizeof(T); }

template <typename T>
__global__ void __launch_bounds__(kXSeg) k_line_blocks_x(LevelV<T> L, int colour) {
  griddep_wait();
  extern __shared__ __align__(16) unsigned char xsm_raw[];
  T* sd = reinterpret_cast<T*>(xsm_raw);
  T* sm = sd + kXPad;
  T* si = sm + kXPad;
  T* sc = si + kXPad;
  const LineGeo g = line_geo<0>(L);
  const int q = 2 * blockIdx.y + colour + 1;
  const int k_base = blockIdx.x * kXPts + 1;      // first point of the segment
  const int o_base = q * g.ls + k_base;
  const T* __restrict__ mu = L.LF[0][LF_MU];
  const T* __restrict__ iu = L.LF[0][LF_IU];
  const T* __restrict__ ca = L.LF[0][LF_CA];
  T* G = L.r;
  const int npts = min(kXPts, g.n - k_base + 1);
  for (int i = threadIdx.x; i < npts; i += kXSeg) {
    const int p = i + i / kLineM, o = o_base + i;
    sd[p] = G[o];
    sm[p] = mu[o];
    si[p] = iu[o];
    sc[p] = ca[o];
  }
  __syncthreads();
  const int j = threadIdx.x;
  const int bb = blockIdx.x * kXSeg + j;
  const int k0 = bb * kLineM + 1;
  const int len = min(kLineM - 1, g.n - k0 + 1);
  if (len > 0) {
    const int pb = j * (kLineM + 1);
    T gfirst, glast;
    block_subst<T>(
        len,
        [&](int e, T& d, T& m, T& iv, T& c) {
          d = sd[pb + e];
          m = sm[pb + e];
          iv = si[pb + e];
          c = sc[pb + e];
        },
        [&](int e, T v) { sd[pb + e] = v; }, gfirst, glast);
    if (k0 + len <= g.n && len == kLineM - 1) {
      const int os = q * g.ls + k0 + len;
      L.SP[0][SP_RL][q * L.spp[0] + bb] = fma(L.W[os], glast, sd[pb + len]);
    }
    if (bb > 0) L.SP[0][SP_GF][q * L.spp[0] + bb - 1] = gfirst;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < npts; i += kXSeg)
    if ((i + 1) % kLineM != 0) G[o_base + i] = sd[i + i / kLineM];
}

// The separators' two-level substitution (line_sep_serial states the
// operations): one thread per group of a line, several lines per thread
// block; each thread substitutes its group from a zero carry, one thread
// per line runs the carries through the groups in shared memory, and each
// thread then fixes up its group.  The right-hand sides come from the
// compact slots the block solves filled.
constexpr int kSepThreads = 256;   // at most: 64 where a line has no more groups
constexpr int kSepGroup = 16;   // separators per group held in registers

template <typename T, int DIR>
__global__ void __launch_bounds__(kSepThreads) k_line_seps(LevelV<T> L, int colour, int ngroups,
                                                           T* __restrict__ xo) {
  griddep_wait();
  __shared__ T s_end[kSepThreads], s_pq[kSepThreads], s_c[kSepThreads];
  const int tid = threadIdx.x;
  const LineGeo g = line_geo<DIR>(L);
  const int lpb = int(blockDim.x) / ngroups;           // lines per block
  const int l = tid / ngroups, gi = tid - l * ngroups;
  const int li = blockIdx.x * lpb + l;
  const bool act = l < lpb && li < line_count(g.nl, colour);
  const int nsep = g.n / kLineM, gl = L.sgl[DIR];
  const int t0 = gi * gl, t1 = min(t0 + gl, nsep);
  const int q = 2 * li + colour + 1;
  const int sp = q * L.spp[DIR];
  const T* __restrict__ mu = L.SP[DIR][SP_MU] + sp;
  const T* __restrict__ iu = L.SP[DIR][SP_IU] + sp;
  const T* __restrict__ ca = L.SP[DIR][SP_CA] + sp;
  const T* __restrict__ an = L.SP[DIR][SP_AN] + sp;
  const T* __restrict__ P = L.SP[DIR][SP_P] + sp;
  const T* __restrict__ Q = L.SP[DIR][SP_Q] + sp;
  const T* __restrict__ gf = L.SP[DIR][SP_GF] + sp;
  T* h = L.SP[DIR][SP_RL] + sp;
  // forward partial substitution of the group (groups of kSepGroup: every
  // load of a phase is issued before its substitution starts)
  constexpr int GL = kSepGroup;
  const bool regs = gl == GL;
  const int len = t1 - t0;
  T hv[GL];
  T yh = T(0);
  if (act) {
    if (regs) {
      T mv[GL], rv[GL];
#pragma unroll
      for (int u = 0; u < GL; ++u)
        if (u < len) {
          mv[u] = mu[t0 + u];
          rv[u] = fma(an[t0 + u], gf[t0 + u], h[t0 + u]);
        }
#pragma unroll
      for (int u = 0; u < GL; ++u)
        if (u < len) {
          yh = fma(mv[u], yh, rv[u]);
          hv[u] = yh;
        }
    } else {
      for (int t = t0; t < t1; ++t) {
        yh = fma(mu[t], yh, fma(an[t], gf[t], h[t]));
        h[t] = yh;
      }
    }
    s_end[tid] = yh;
    s_pq[tid] = P[t1 - 1];
  }
  __syncthreads();
  if (act && gi == 0) {
    T c = T(0);
    for (int k = 0; k < ngroups; ++k) {
      const int j = l * ngroups + k;
      const T cg = c;
      s_c[j] = cg;
      c = fma(s_pq[j], cg, s_end[j]);
    }
  }
  __syncthreads();
  // fix-up, scaling and backward partial substitution of the group
  if (act) {
    const T cg = s_c[tid];
    T xh = T(0);
    if (regs) {
      T pv[GL], iv[GL], cv[GL];
#pragma unroll
      for (int u = 0; u < GL; ++u)
        if (u < len) {
          pv[u] = P[t0 + u];
          iv[u] = iu[t0 + u];
          cv[u] = ca[t0 + u];
        }
#pragma unroll
      for (int u = GL - 1; u >= 0; --u)
        if (u < len) {
          xh = fma(cv[u], xh, fma(pv[u], cg, hv[u]) * iv[u]);
          hv[u] = xh;
        }
    } else {
      for (int t = t1 - 1; t >= t0; --t) {
        xh = fma(ca[t], xh, fma(P[t], cg, h[t]) * iu[t]);
        h[t] = xh;
      }
    }
    s_end[tid] = xh;
    s_pq[tid] = Q[t0];
  }
  __syncthreads();
  if (act && gi == 0) {
    T e = T(0);
    for (int k = ngroups - 1; k >= 0; --k) {
      const int j = l * ngroups + k;
      s_c[j] = e;
      e = fma(s_pq[j], e, s_end[j]);
    }
  }
  __syncthreads();
  if (act) {
    const T e = s_c[tid];
    const int base = q * g.ls;
    if (regs) {
#pragma unroll
      for (int u = 0; u < GL; ++u)
        if (u < len) xo[base + (t0 + u + 1) * kLineM * g.es] = fma(Q[t0 + u], e, hv[u]);
    } else {
      for (int t = t0; t < t1; ++t) xo[base + (t + 1) * kLineM * g.es] = fma(Q[t], e, h[t]);
    }
  }
}

template <typename T, int DIR>
__global__ void __launch_bounds__(kPT) k_line_final(LevelV<T> L, int colour,
                                                    T* __restrict__ xo) {
  griddep_wait();
  const LineGeo g = line_geo<DIR>(L);
  for_colour_points<DIR>(g, colour, [&](int q, int k) {
    if (k % kLineM != 0) line_final<T, DIR>(L, g, q, k, xo);
  });
}

// ---------------------------------------------------------------------------
// One (direction, colour) step in one kernel: a thread block takes whole lines
// from the right-hand sides to the final update.
//
// What bounds it.  The four launches above move the scratch plane in and out
// of memory three times, and on the levels below a few hundred points a side
// their time is launches and the latency of the separators' chain (17 us a
// launch on every level: one thread carried a group's right-hand sides,
// forward substitution, fix-up, scaling, back substitution and update, 96
// dependent FP64 instructions at 64 cycles each and more where two warps
// shared an SM quarter, on as few SMs as 256-thread blocks of groups fill;
// 13 us with 64-thread blocks).
// Here the line stays in shared memory, and only the two substitutions of
// the separators are chains (16 steps a group); their right-hand sides,
// fix-ups, scalings and updates are one separator per thread.  Every value
// is computed by the same operations as in the four kernels.
//
// C lines per block: one x-line, whose factors are staged too (threads solve
// blocks of 16 points, so unstaged loads would be 128 bytes apart); or up to
// eight columns of one colour, whose factors lie side by side.  Position i of
// line c is at (i + i / 16) * C + c: the padding spreads the blocks over the
// banks.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void step_copy(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                   static_cast<unsigned>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void step_copy(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   static_cast<unsigned>(__cvta_generic_to_shared(dst))),
               "l"(src)
               : "memory");
}

template <typename T, int DIR, int C>
struct StepSmem {
  int g, nb, ng;   // elements of a line plane, of the block arrays, of the group arrays
  __host__ __device__ StepSmem(int n, int sgl) {
    g = (n + n / kLineM + 1) * C;
    nb = (n / kLineM + 1) * C;
    ng = (n / kLineM / sgl + 1) * C;
  }
  // line plane (x-lines: and three factor planes), first / last solutions,
  // separators' values and multipliers, groups' end values, products, carries
  __host__ __device__ size_t bytes() const {
    return sizeof(T) * (size_t(g) * (DIR == 0 ? 4 : 1) + 4 * size_t(nb) + 3 * size_t(ng));
  }
};

template <typename T, int DIR, bool NINE, int C, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_line_step(LevelV<T> L, int colour, const T* __restrict__ xs,
                                                  T* xo) {
  extern __shared__ __align__(16) unsigned char step_raw[];
  const LineGeo g = line_geo<DIR>(L);
  const int n = g.n, nsep = n / kLineM, nb = nsep + 1, gl = L.sgl[DIR], ng = cdiv(nsep, gl);
  const StepSmem<T, DIR, C> m(n, gl);
  T* const G = reinterpret_cast<T*>(step_raw);
  T* const FM = G + m.g;                                  // x-lines: mu, iu, ca
  T* const gfirst = G + (DIR == 0 ? 4 : 1) * m.g;
  T* const glast = gfirst + m.nb;
  T* const H = glast + m.nb;                              // separators
  T* const M = H + m.nb;
  T* const gend = M + m.nb;                               // groups
  T* const gpq = gend + m.ng;
  T* const gc = gpq + m.ng;
  const int l0 = blockIdx.x * C;                          // first line of the colour
  const int lines = min(C, line_count(g.nl, colour) - l0);
  const T* A = line_coupling<DIR>(L);
  auto line = [&](int c) { return 2 * (l0 + c) + colour + 1; };
  auto at = [](int i, int c) { return (i + i / kLineM) * C + c; };
  const T* __restrict__ mu = L.LF[DIR][LF_MU];
  const T* __restrict__ iu = L.LF[DIR][LF_IU];
  const T* __restrict__ ca = L.LF[DIR][LF_CA];
  if (DIR == 0) {
    // (constant since the setup)
    const int f = line_fbase<DIR>(L, line(0)) + 1;
    for (int i = threadIdx.x; i < n; i += NT) {
      const int p = at(i, 0);
      step_copy(FM + p, mu + f + i);
      step_copy(FM + m.g + p, iu + f + i);
      step_copy(FM + 2 * m.g + p, ca + f + i);
    }
  }
  griddep_wait();
  // U points' loads in flight at once: one by one, a line's rows of loads
  // took 100 us on 1024 lines of 2047 points
  constexpr int U = NINE ? 2 : 4;
  for (int e0 = threadIdx.x; e0 < n * C; e0 += U * NT) {
    T d[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * NT, i = e / C, c = e - i * C;
      if (e < n * C && c < lines) d[u] = line_rhs<T, DIR, NINE>(L, xs, line(c) * g.ls + (i + 1) * g.es);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = e0 + u * NT, i = e / C, c = e - i * C;
      if (e < n * C && c < lines) G[at(i, c)] = d[u];
    }
  }
  if (DIR == 0) asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  // block solves (block_subst, with the forward values in shared memory and
  // few registers, so that two or three blocks share an SM)
  constexpr int M1 = kLineM - 1;
  for (int e = threadIdx.x; e < nb * C; e += NT) {
    const int bb = e / C, c = e - bb * C;
    const int len = min(M1, n - bb * kLineM);
    T first = T(0), last = T(0);
    if (c < lines && len > 0) {
      const int p0 = at(bb * kLineM, c);
      const int f0 = line_fbase<DIR>(L, line(c)) + (bb * kLineM + 1) * g.fes;
      auto factor = [&](const T* __restrict__ global, int plane, int k) {
        return DIR == 0 ? FM[plane * m.g + p0 + k * C] : global[f0 + k * g.fes];
      };
      {
        T mv[M1];
#pragma unroll
        for (int k = 0; k < M1; ++k)
          if (k < len) mv[k] = factor(mu, 0, k);
        T prev = T(0);
#pragma unroll
        for (int k = 0; k < M1; ++k)
          if (k < len) {
            prev = fma(mv[k], prev, G[p0 + k * C]);
            G[p0 + k * C] = prev;
          }
      }
      T next = T(0);
      constexpr int HB = (M1 + 1) / 2;
#pragma unroll
      for (int h = M1 - 1; h >= 0; h -= HB) {
        T iv[HB], cv[HB];
#pragma unroll
        for (int k = 0; k < HB; ++k)
          if (h - k >= 0 && h - k < len) {
            iv[k] = factor(iu, 1, h - k);
            cv[k] = factor(ca, 2, h - k);
          }
#pragma unroll
        for (int k = 0; k < HB; ++k)
          if (h - k >= 0 && h - k < len) {
            next = fma(cv[k], next, G[p0 + (h - k) * C] * iv[k]);
            if (h - k == len - 1) last = next;
            G[p0 + (h - k) * C] = next;
          }
      }
      first = next;
    }
    gfirst[e] = first;
    glast[e] = last;
  }
  __syncthreads();
  if (nsep > 0) {
    // separators' right-hand sides; the forward multipliers
    for (int e = threadIdx.x; e < nsep * C; e += NT) {
      const int t = e / C, c = e - t * C;
      if (c >= lines) continue;
      const int q = line(c), sp = q * L.spp[DIR] + t, i = (t + 1) * kLineM - 1;
      const T r = fma(A[q * g.ls + (i + 1) * g.es], glast[e], G[at(i, c)]);
      H[e] = fma(L.SP[DIR][SP_AN][sp], gfirst[e + C], r);
      M[e] = L.SP[DIR][SP_MU][sp];
    }
    __syncthreads();
    // forward within the groups
    for (int e = threadIdx.x; e < ng * C; e += NT) {
      const int gi = e / C, c = e - gi * C;
      if (c >= lines) continue;
      const int t1 = min((gi + 1) * gl, nsep);
      T yh = T(0);
      for (int t = gi * gl; t < t1; ++t) {
        yh = fma(M[t * C + c], yh, H[t * C + c]);
        H[t * C + c] = yh;
      }
      gend[e] = yh;
      gpq[e] = L.SP[DIR][SP_P][line(c) * L.spp[DIR] + t1 - 1];
    }
    __syncthreads();
    for (int c = threadIdx.x; c < lines; c += NT) {
      T v = T(0);
      for (int k = 0; k < ng; ++k) {
        gc[k * C + c] = v;
        v = fma(gpq[k * C + c], v, gend[k * C + c]);
      }
    }
    __syncthreads();
    // fix-up and scaling; the backward multipliers
    for (int e = threadIdx.x; e < nsep * C; e += NT) {
      const int t = e / C, c = e - t * C;
      if (c >= lines) continue;
      const int sp = line(c) * L.spp[DIR] + t;
      H[e] = fma(L.SP[DIR][SP_P][sp], gc[t / gl * C + c], H[e]) * L.SP[DIR][SP_IU][sp];
      M[e] = L.SP[DIR][SP_CA][sp];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < ng * C; e += NT) {
      const int gi = e / C, c = e - gi * C;
      if (c >= lines) continue;
      const int t0 = gi * gl, t1 = min(t0 + gl, nsep);
      T xh = T(0);
      for (int t = t1 - 1; t >= t0; --t) {
        xh = fma(M[t * C + c], xh, H[t * C + c]);
        H[t * C + c] = xh;
      }
      gend[e] = xh;
      gpq[e] = L.SP[DIR][SP_Q][line(c) * L.spp[DIR] + t0];
    }
    __syncthreads();
    for (int c = threadIdx.x; c < lines; c += NT) {
      T v = T(0);
      for (int k = ng - 1; k >= 0; --k) {
        gc[k * C + c] = v;
        v = fma(gpq[k * C + c], v, gend[k * C + c]);
      }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nsep * C; e += NT) {
      const int t = e / C, c = e - t * C;
      if (c >= lines) continue;
      H[e] = fma(L.SP[DIR][SP_Q][line(c) * L.spp[DIR] + t], gc[t / gl * C + c], H[e]);
    }
    __syncthreads();
  }
  // final update (line_final): a block's g plus the spikes times its
  // separators, 0 where the line ends
  const T* __restrict__ lv = L.LF[DIR][LF_V];
  const T* __restrict__ lw = L.LF[DIR][LF_W];
  for (int e0 = threadIdx.x; e0 < n * C; e0 += 4 * NT) {
    T vv[4], wv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = e0 + u * NT, i = e / C, c = e - i * C;
      if (e < n * C && c < lines) {
        const int f = line_fbase<DIR>(L, line(c)) + (i + 1) * g.fes;
        vv[u] = lv[f];
        wv[u] = lw[f];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = e0 + u * NT, i = e / C, c = e - i * C;
      if (e >= n * C || c >= lines) continue;
      const int bb = i / kLineM;
      T v;
      if ((i + 1) % kLineM == 0) {
        v = H[bb * C + c];
      } else {
        const T xl = bb > 0 ? H[(bb - 1) * C + c] : T(0), xr = bb < nsep ? H[bb * C + c] : T(0);
        v = fma(wv[u], xr, fma(vv[u], xl, G[at(i, c)]));
      }
      xo[line(c) * g.ls + (i + 1) * g.es] = v;
    }
  }
}

// Shared memory a step may take: two blocks and more per SM.
constexpr size_t kStepSmem = 110 * 1024;

template <typename T, int DIR, bool NINE, int C>
bool launch_line_step_c(const LevelV<T>& L, int colour, const T* xs, T* xo, cudaStream_t s) {
  constexpr int NT = 256, MINB = DIR == 0 ? 3 : (C <= 2 ? 4 : 3);
  const LineGeo g = line_geo<DIR>(L);
  const size_t smem = StepSmem<T, DIR, C>(g.n, L.sgl[DIR]).bytes();
  if (smem > kStepSmem) return false;
  if (!use_shared(k_line_step<T, DIR, NINE, C, NT, MINB>, kStepSmem)) return false;
  launch_pdl(k_line_step<T, DIR, NINE, C, NT, MINB>, dim3(cdiv(line_count(g.nl, colour), C)), dim3(NT), smem, s, L,
             colour, xs, xo);
  count_launch();
  return true;
}

// The fused step on levels of at most kStepPoints points; above that the four
// kernels' wider parallelism wins (2047^2, FP64, per step: x-lines 73 us in
// four launches against 71 fused, y-lines 69 against 116, whose columns keep
// half of every sector of the planes idle in each of few large blocks; on
// 511^2 and below 20 to 30 us in four launches against 10 to 20 fused;
// alternating V(2,1) solve of 2047^2 with the line at 5 M, 1.2 M and 300 k
// points: 31.0, 27.9, 27.0 ms of kernels).  Columns: as many per block as
// still give 64 blocks (128: 31.3 ms, 64: 30.9, 32: 31.8, all levels fused).
constexpr long kStepPoints = 300000;
constexpr int kStepBlocks = 64;
template <typename T, int DIR, bool NINE>
bool launch_line_step(const LevelV<T>& L, int colour, const T* xs, T* xo, cudaStream_t s) {
  if (long(L.nx) * L.ny > kStepPoints) return false;
  const int nlc = line_count(line_geo<DIR>(L).nl, colour);
  if constexpr (DIR == 0) {
    return launch_line_step_c<T, 0, NINE, 1>(L, colour, xs, xo, s);
  } else {
    return (nlc >= 8 * kStepBlocks && launch_line_step_c<T, 1, NINE, 8>(L, colour, xs, xo, s)) ||
           (nlc >= 4 * kStepBlocks && launch_line_step_c<T, 1, NINE, 4>(L, colour, xs, xo, s)) ||
           (nlc >= 2 * kStepBlocks && launch_line_step_c<T, 1, NINE, 2>(L, colour, xs, xo, s)) ||
           launch_line_step_c<T, 1, NINE, 1>(L, colour, xs, xo, s);
  }
}

// ---------------------------------------------------------------------------
// Setup: factors of every line (both colours), computed in FP64 and stored
// in the level's precision.
// ---------------------------------------------------------------------------

// Per block: LU of the block's tridiagonal matrix (diagonal C, off-diagonals
// -a) and its responses v = T^{-1} (a_first e_first), w = T^{-1} (a_next e_last)
// to unit values of the separators on either side (a_first couples the
// block's first point to the point before it, a_next its last point to the
// point after it; both are 0 at the ends of the line).
template <typename T, int DIR>
__global__ void __launch_bounds__(kBT) k_line_factor_blocks(LevelV<T> L, int* derr) {
  const LineGeo g = line_geo<DIR>(L);
  const int nb = g.n / kLineM + 1;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nb * g.nl) return;
  const int q = t / nb + 1, bb = t % nb;
  const int k0 = bb * kLineM + 1;
  const int len = min(kLineM - 1, g.n - k0 + 1);
  if (len <= 0) return;
  const T* A = line_coupling<DIR>(L);
  const int o0 = q * g.ls + k0 * g.es;
  const int f0 = line_fbase<DIR>(L, q) + k0 * g.fes;
  double iu[kLineM - 1], ca[kLineM - 1], mu[kLineM - 1];
  double up = 1.0;
  bool bad = false;
#pragma unroll
  for (int e = 0; e < kLineM - 1; ++e) {
    if (e < len) {
      const int o = o0 + e * g.es;
      const double a = double(A[o]), c = double(L.C[o]);
      const double m = e ? a / up : 0.0;
      const double u = c - m * a;
      if (!(u > 0.0) || !(u < INFINITY)) bad = true;
      mu[e] = m;
      iu[e] = 1.0 / u;
      if (e) ca[e - 1] = a * iu[e - 1];
      up = u;
    }
  }
  const double a_first = double(A[o0]);
  const double a_next = double(A[o0 + len * g.es]);
  double yv[kLineM - 1];
  double prev = a_first;
#pragma unroll
  for (int e = 0; e < kLineM - 1; ++e) {
    if (e < len) {
      if (e) prev = mu[e] * prev;
      yv[e] = prev;
    }
  }
  double vn = 0.0, wn = 0.0;
#pragma unroll
  for (int e = kLineM - 2; e >= 0; --e) {
    if (e < len) {
      const int f = f0 + e * g.fes;
      const double cae = e == len - 1 ? 0.0 : ca[e];
      vn = yv[e] * iu[e] + cae * vn;
      wn = (e == len - 1 ? a_next * iu[e] : 0.0) + cae * wn;
      L.LF[DIR][LF_MU][f] = T(mu[e]);
      L.LF[DIR][LF_IU][f] = T(iu[e]);
      L.LF[DIR][LF_CA][f] = T(cae);
      L.LF[DIR][LF_V][f] = T(vn);
      L.LF[DIR][LF_W][f] = T(wn);
    }
  }
  if (bad) atomicOr(derr, DEV_BADLINE);
}

// Per line: the Schur complement on the separators.  With the interior
// points written as g + v x_left + w x_right, the equation of separator s is
//   (C_s - a_s w_{s-1} - a_{s+1} v_{s+1}) x_s - a_s v_{s-1} x_prev
//     - a_{s+1} w_{s+1} x_next = d_s + a_s g_{s-1} + a_{s+1} g_{s+1},
// a tridiagonal system over the separators of the line, factored here.
template <typename T, int DIR>
__global__ void __launch_bounds__(kBT) k_line_factor_seps(LevelV<T> L, int* derr) {
  const LineGeo g = line_geo<DIR>(L);
  const int q = blockIdx.x * blockDim.x + threadIdx.x + 1;
  if (q > g.nl) return;
  const int nsep = g.n / kLineM;
  const T* A = line_coupling<DIR>(L);
  const T* V = L.LF[DIR][LF_V];
  const T* W = L.LF[DIR][LF_W];
  double up = 1.0, uprev_coupling = 0.0;
  bool bad = false;
  for (int t = 0; t < nsep; ++t) {
    const int os = q * g.ls + (t + 1) * kLineM * g.es;
    const int fs = line_fbase<DIR>(L, q) + (t + 1) * kLineM * g.fes;
    const double as = double(A[os]), an = double(A[os + g.es]);
    const double d = double(L.C[os]) - as * double(W[fs - g.fes]) - an * double(V[fs + g.fes]);
    const double lo = as * double(V[fs - g.fes]);   // coupling to the previous separator
    const double hi = an * double(W[fs + g.fes]);   // coupling to the next separator
    const double m = t ? lo / up : 0.0;
    const double u = d - m * uprev_coupling;
    if (!(u > 0.0) || !(u < INFINITY)) bad = true;
    const int c = q * L.spp[DIR] + t;
    L.SP[DIR][SP_MU][c] = T(m);
    L.SP[DIR][SP_IU][c] = T(1.0 / u);
    L.SP[DIR][SP_CA][c] = T(hi / u);
    L.SP[DIR][SP_AN][c] = A[os + g.es];
    up = u;
    uprev_coupling = hi;
  }
  // products of the stored multipliers over each group: P from the group's
  // start to t, Q from t to the group's end
  const int gl = L.sgl[DIR];
  T* mu = L.SP[DIR][SP_MU] + q * L.spp[DIR];
  T* ca = L.SP[DIR][SP_CA] + q * L.spp[DIR];
  T* P = L.SP[DIR][SP_P] + q * L.spp[DIR];
  T* Q = L.SP[DIR][SP_Q] + q * L.spp[DIR];
  double pr = 1.0;
  for (int t = 0; t < nsep; ++t) {
    pr = (t % gl == 0 ? 1.0 : pr) * double(mu[t]);
    P[t] = T(pr);
  }
  for (int t = nsep - 1; t >= 0; --t) {
    pr = (t == nsep - 1 || (t + 1) % gl == 0 ? 1.0 : pr) * double(ca[t]);
    Q[t] = T(pr);
  }
  if (bad) atomicOr(derr, DEV_BADLINE);
}

int grid_y(int slow) { return slow < 65535 ? slow : 65535; }

template <typename T, int DIR, bool NINE>
void line_step(const LevelV<T>& L, int colour, const T* xs, T* xo, cudaStream_t s) {
  const LineGeo g = line_geo<DIR>(L);
  const int nlc = line_count(g.nl, colour);
  if (nlc <= 0) return;
  if (launch_line_step<T, DIR, NINE>(L, colour, xs, xo, s)) return;
  const int nb = g.n / kLineM + 1;
  {
    const int fast = DIR == 0 ? g.n : nlc, slow = DIR == 0 ? nlc : g.n;
    launch_pdl(k_line_rhs<T, DIR, NINE>, dim3(cdiv(fast, kPT), grid_y(slow)), dim3(kPT), 0, s, L, colour, xs);
  }
  if (DIR == 0) {
    launch_pdl(k_line_blocks_x<T>, dim3(cdiv(g.n, kXPts), nlc), dim3(kXSeg), xblocks_smem<T>(), s, L, colour);
  } else {
    const int fast = nlc, slow = nb;
    launch_pdl(k_line_blocks<T, DIR>, dim3(cdiv(fast, kBT), grid_y(slow)), dim3(kBT), 0, s, L, colour);
  }
  if (g.n >= kLineM) {
    // two warps a block: 256-thread blocks of 1024 lines' groups covered 32 SMs
    const int nsep = g.n / kLineM, ngroups = cdiv(nsep, L.sgl[DIR]);
    const int nt = ngroups <= 64 ? 64 : kSepThreads;
    launch_pdl(k_line_seps<T, DIR>, dim3(cdiv(nlc, nt / ngroups)), dim3(nt), 0, s, L, colour, ngroups, xo);
  }
  {
    const int fast = DIR == 0 ? g.n : nlc, slow = DIR == 0 ? nlc : g.n;
    launch_pdl(k_line_final<T, DIR>, dim3(cdiv(fast, kPT), grid_y(slow)), dim3(kPT), 0, s, L, colour, xo);
  }
  count_launch(g.n >= kLineM ? 4 : 3);
}

}  // namespace

template <typename T>
int launch_line_factor(const LevelV<T>& L, int smoother, int* derr, cudaStream_t s) {
  if (!allow_shared(k_line_blocks_x<T>, xblocks_smem<T>())) return BMG_ECUDA;
  auto one = [&](auto dir_tag) {
    constexpr int DIR = decltype(dir_tag)::value;
    const LineGeo g = line_geo<DIR>(L);
    const int nb = g.n / kLineM + 1;
    k_line_factor_blocks<T, DIR><<<cdiv(nb * g.nl, kBT), kBT, 0, s>>>(L, derr);
    k_line_factor_seps<T, DIR><<<cdiv(g.nl, kBT), kBT, 0, s>>>(L, derr);
    count_launch(2);
  };
  if (smoother == BMG_SMOOTH_XLINE || smoother == BMG_SMOOTH_ALTLINE)
    one(std::integral_constant<int, 0>{});
  if (smoother == BMG_SMOOTH_YLINE || smoother == BMG_SMOOTH_ALTLINE)
    one(std::integral_constant<int, 1>{});
  return cudaGetLastError() == cudaSuccess ? 0 : BMG_ECUDA;
}

template <typename T>
void launch_line_sweep(const LevelV<T>& L, bool nine, int smoother, bool reverse, const T* xin,
                       T* xout, cudaStream_t s) {
  int dir[4], colour[4];
  const int n = line_steps(smoother, reverse, dir, colour);
  for (int k = 0; k < n; ++k) {
    // The first step reads the neighbouring lines from xin; every later one
    // from xout, which holds all lines the earlier steps solved.
    const T* xs = k == 0 ? xin : xout;
    if (dir[k] == 0) {
      if (nine)
        line_step<T, 0, true>(L, colour[k], xs, xout, s);
      else
        line_step<T, 0, false>(L, colour[k], xs, xout, s);
    } else {
      if (nine)
        line_step<T, 1, true>(L, colour[k], xs, xout, s);
      else
        line_step<T, 1, false>(L, colour[k], xs, xout, s);
    }
  }
}

template int launch_line_factor<double>(const LevelV<double>&, int, int*, cudaStream_t);
template int launch_line_factor<float>(const LevelV<float>&, int, int*, cudaStream_t);
template void launch_line_sweep<double>(const LevelV<double>&, bool, int, bool, const double*,
                                        double*, cudaStream_t);
template void launch_line_sweep<float>(const LevelV<float>&, bool, int, bool, const float*, float*,
                                       cudaStream_t);

}  // namespace bmg
