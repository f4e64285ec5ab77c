// Launches of the fused V-cycle legs of one level (bmg_legs.cuh).
#include "bmg_legs.cuh"

namespace bmg {

namespace {

inline int cdiv(int a, int b) { return (a + b - 1) / b; }

// Legs of at most this many (8 x 8) blocks let the next kernel's blocks start
// early (griddep_launch; in every leg it cost 511^2 7 %: the 32 x 16 tiles'
// successors hold the shared memory they need).
constexpr unsigned kEarly = 152;

template <typename T, bool NINE, int NS, bool ZERO, int TX, int TY, int NT>
__global__ void __launch_bounds__(NT) k_down(LevelV<T> F, const T* __restrict__ xin,
                                             T* __restrict__ xout, LevelV<T> Cc) {
  extern __shared__ __align__(16) unsigned char leg_smem[];
  T* sm = reinterpret_cast<T*>(leg_smem);
  T pw[8];
  down_constants<T, NINE, NS, TX, TY, NT>(F, Cc, sm, blockIdx.x, blockIdx.y, pw);
  griddep_wait();
  if (TX * TY <= 64 && gridDim.x * gridDim.y <= kEarly) griddep_launch();
  down_tile<T, NINE, NS, ZERO, TX, TY, NT>(F, xin, xout, Cc, sm, blockIdx.x, blockIdx.y, pw);
}

template <typename T, bool NINE, int TX, int TY, int NT, bool NRM>
__global__ void __launch_bounds__(NT) k_up(LevelV<T> F, const T* __restrict__ xin,
                                           const T* __restrict__ xc, T* __restrict__ xout,
                                           T* __restrict__ xnext, double* __restrict__ partials) {
  extern __shared__ __align__(16) unsigned char leg_smem[];
  T* sm = reinterpret_cast<T*>(leg_smem);
  T w[8];
  up_constants<T, NINE, TX, TY, NT, NRM>(F, sm, blockIdx.x, blockIdx.y, w);
  griddep_wait();
  if (TX * TY <= 64 && gridDim.x * gridDim.y <= kEarly) griddep_launch();
  const double a =
      up_tile<T, NINE, TX, TY, NT, NRM>(F, xin, xc, xout, xnext, sm, blockIdx.x, blockIdx.y, w);
  if (NRM && threadIdx.x == 0) partials[blockIdx.y * gridDim.x + blockIdx.x] = a;
}

template <typename T, bool NINE, int NS, bool ZERO, int TX, int TY, int NT>
void down_shape(const LevelV<T>& F, const T* xin, T* xout, const LevelV<T>& Cc, cudaStream_t s) {
  constexpr size_t smem = DownLeg<T, NINE, NS, TX, TY>::SMEM;
  launch_pdl(k_down<T, NINE, NS, ZERO, TX, TY, NT>, dim3(cdiv(F.nx, TX), cdiv(F.ny, TY)), dim3(NT), smem,
             s, F, xin, xout, Cc);
}

template <typename T, bool NINE, int TX, int TY, int NT, bool NRM>
void up_shape(const LevelV<T>& F, const T* xin, const T* xc, T* xout, T* xnext, double* partials,
              cudaStream_t s) {
  constexpr size_t smem = UpLeg<T, NINE, TX, TY, NRM>::SMEM;
  launch_pdl(k_up<T, NINE, TX, TY, NT, NRM>, dim3(cdiv(F.nx, TX), cdiv(F.ny, TY)), dim3(NT), smem, s, F,
             xin, xc, xout, xnext, partials);
}

template <typename T, int TX, int TY, int NT>
void down_kind(const LevelV<T>& F, bool nine, int ns, bool zero, const T* xin, T* xout,
               const LevelV<T>& Cc, cudaStream_t s) {
#define BMG_DOWN(NINE, NS)                                                  \
  do {                                                                      \
    if (zero)                                                               \
      down_shape<T, NINE, NS, true, TX, TY, NT>(F, xin, xout, Cc, s);       \
    else                                                                    \
      down_shape<T, NINE, NS, false, TX, TY, NT>(F, xin, xout, Cc, s);      \
  } while (0)
  if (nine && ns == 2) BMG_DOWN(true, 2);
  else if (nine) BMG_DOWN(true, 1);
  else if (ns == 2) BMG_DOWN(false, 2);
  else BMG_DOWN(false, 1);
#undef BMG_DOWN
}

template <typename T, int TX, int TY, int NT>
void up_kind(const LevelV<T>& F, bool nine, const T* xin, const T* xc, T* xout, T* xnext,
             double* partials, cudaStream_t s) {
  if (nine)
    up_shape<T, true, TX, TY, NT, false>(F, xin, xc, xout, nullptr, nullptr, s);
  else if (partials)
    up_shape<T, false, TX, TY, NT, true>(F, xin, xc, xout, xnext, partials, s);
  else
    up_shape<T, false, TX, TY, NT, false>(F, xin, xc, xout, nullptr, nullptr, s);
}

// The shared memory of a shape's kernels, on the current device.
template <typename T, bool NINE, int TX, int TY, int NT>
bool shape_ready() {
  using D1 = DownLeg<T, NINE, 1, TX, TY>;
  using D2 = DownLeg<T, NINE, 2, TX, TY>;
  bool ok = use_shared(k_down<T, NINE, 1, false, TX, TY, NT>, D1::SMEM) &&
            use_shared(k_down<T, NINE, 1, true, TX, TY, NT>, D1::SMEM) &&
            use_shared(k_down<T, NINE, 2, false, TX, TY, NT>, D2::SMEM) &&
            use_shared(k_down<T, NINE, 2, true, TX, TY, NT>, D2::SMEM) &&
            use_shared(k_up<T, NINE, TX, TY, NT, false>, UpLeg<T, NINE, TX, TY, false>::SMEM);
  if constexpr (!NINE) ok = ok && use_shared(k_up<T, false, TX, TY, NT, true>, UpLeg<T, false, TX, TY, true>::SMEM);
  return ok;
}

}  // namespace

// Which levels take the fused legs, and with which tile.  Every leg is a
// chain of phases whose length does not depend on the tile, so as long as
// the tiles do not fill the GPU (304: two for each of its 152 SMs) the
// smallest are the best (fewest warps per FP64 phase); past that the halo's
// redundant work decides.  The limits count tiles, and were measured on
// square grids of 2^m - 1 points a side only: each lies somewhere between
// the tile counts of two such levels.  Measured (us per V-cycle, FP64 unless
// said otherwise):
//  * 8 x 8 up to 304 tiles (two per SM): 127^2 52.9 against 53.9 with 16 x 8,
//    255^2 66.5 against 67.2; up to 1100 tiles 255^2 takes 68.0;
//  * 16 x 8 up to 320 tiles: 511^2 99.0; up to 608, 102.8 (its 255^2 level
//    prefers 32 x 16);
//  * 32 x 16 beyond: on 9-point levels the two sweeps' halo work costs more
//    FP64 time than the launches from about 500 tiles on (1023^2, whose 511^2
//    level has 512: 189.2 without, 196.1 with; FP32 1023^2: 117 with, 122
//    without 511^2; FP32 4095^2, whose 1023^2 level has 2048: 894.7 without,
//    899.8 with), red-black legs grow less (511^2: 94.8 with the finest
//    level's legs, 99.2 without; FP32 1023^2: 115.9 with, 122.2 without).
// Launched one operation at a time the same cycles take 106 (255^2), 131
// (511^2), in FP32 82 and 100.
enum { LEG_16x8 = 1, LEG_32x16, LEG_8x8 };

template <typename T>
bool leg_ready(int shape, bool nine) {
  switch (shape) {
    case LEG_8x8: return nine ? shape_ready<T, true, 8, 8, 128>() : shape_ready<T, false, 8, 8, 128>();
    case LEG_16x8: return nine ? shape_ready<T, true, 16, 8, 128>() : shape_ready<T, false, 16, 8, 128>();
    case LEG_32x16: return nine ? shape_ready<T, true, 32, 16, 256>() : shape_ready<T, false, 32, 16, 256>();
    default: return false;
  }
}
template bool leg_ready<double>(int, bool);
template bool leg_ready<float>(int, bool);

int leg_shape(int nx, int ny, bool nine, bool fp64) {
  if (cdiv(nx, 8) * cdiv(ny, 8) <= 304) return LEG_8x8;
  if (cdiv(nx, 16) * cdiv(ny, 8) <= 320) return LEG_16x8;
  const int most = fp64 ? (nine ? 320 : 640) : (nine ? 608 : 2100);
  return cdiv(nx, 32) * cdiv(ny, 16) <= most ? LEG_32x16 : 0;
}

int leg_tiles(int shape, int nx, int ny) {
  switch (shape) {
    case LEG_8x8: return cdiv(nx, 8) * cdiv(ny, 8);
    case LEG_16x8: return cdiv(nx, 16) * cdiv(ny, 8);
    case LEG_32x16: return cdiv(nx, 32) * cdiv(ny, 16);
    default: return 0;
  }
}

template <typename T>
void launch_down_leg(const LevelV<T>& F, bool nine, int shape, int ns, bool zero, const T* xin, T* xout,
                     const LevelV<T>& Cc, cudaStream_t s) {
  if (shape == LEG_8x8)
    down_kind<T, 8, 8, 128>(F, nine, ns, zero, xin, xout, Cc, s);
  else if (shape == LEG_16x8)
    down_kind<T, 16, 8, 128>(F, nine, ns, zero, xin, xout, Cc, s);
  else
    down_kind<T, 32, 16, 256>(F, nine, ns, zero, xin, xout, Cc, s);
  count_launch();
}

template <typename T>
void launch_up_leg(const LevelV<T>& F, bool nine, int shape, const T* xin, const T* xc, T* xout, T* xnext,
                   double* partials, cudaStream_t s) {
  if (shape == LEG_8x8)
    up_kind<T, 8, 8, 128>(F, nine, xin, xc, xout, xnext, partials, s);
  else if (shape == LEG_16x8)
    up_kind<T, 16, 8, 128>(F, nine, xin, xc, xout, xnext, partials, s);
  else
    up_kind<T, 32, 16, 256>(F, nine, xin, xc, xout, xnext, partials, s);
  count_launch();
}

template void launch_down_leg<double>(const LevelV<double>&, bool, int, int, bool, const double*, double*,
                                      const LevelV<double>&, cudaStream_t);
template void launch_down_leg<float>(const LevelV<float>&, bool, int, int, bool, const float*, float*,
                                     const LevelV<float>&, cudaStream_t);
template void launch_up_leg<double>(const LevelV<double>&, bool, int, const double*, const double*,
                                    double*, double*, double*, cudaStream_t);
template void launch_up_leg<float>(const LevelV<float>&, bool, int, const float*, const float*, float*,
                                   float*, double*, cudaStream_t);

}  // namespace bmg
