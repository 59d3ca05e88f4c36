// passes_inst.cu -- host launchers of the mesh passes for one FFT-domain side
// N = MOND_N (this file is compiled once per supported size, in parallel).
#include "launch.h"
#include "regpass.cuh"
#include "xreg.cuh"

#ifndef MOND_N
#error "compile with -DMOND_N=<size>"
#endif

namespace {
using namespace passes;
constexpr int N = MOND_N;

template <typename K>
cudaError_t set_smem(K kern, size_t bytes) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

size_t x_smem(int nc) { return sizeof(float2) * (N + (size_t)nc * XCfg<N>::ROWS * XCfg<N>::LP); }
size_t y_smem() { return sizeof(float2) * (N + (size_t)N * YZCfg<N>::P); }
size_t z_smem(int ntiles) { return sizeof(float2) * (2 * N + (size_t)ntiles * N * YZCfg<N>::P); }

template <int MODE>
cudaError_t launch_x(const XArgs& a, cudaStream_t st) {
  const size_t sm = x_smem((MODE == X_RHO || MODE == X_DRHO) ? 1 : 3);
  cudaError_t e = set_smem(k_xpass<N, MODE>, sm);
  if (e != cudaSuccess) return e;
  int64_t nlines = (int64_t)N * N;
  return launch_early(k_xpass<N, MODE>, (unsigned)(nlines / XCfg<N>::L), NTX, sm, st, a, nlines);
}

template <int MODE>
cudaError_t launch_xreg(const XArgs& a, cudaStream_t st) {
  using X = xreg::Geo<N>;
  constexpr size_t sm = xreg::smem_bytes<N, MODE>();
  cudaError_t e = sm > 48 * 1024 ? set_smem(xreg::k_xreg<N, MODE>, sm) : cudaSuccess;
  if (e != cudaSuccess) return e;
  const dim3 grid(N * N / X::LINES, xreg::ncomp_of(MODE) == 3 ? 1 : a.ncomp);
  return launch_early(xreg::k_xreg<N, MODE>, grid, 32 * xreg::WARPS, sm, st, a);
}

template <int MODE>
cudaError_t launch_z(const ZArgs& a, cudaStream_t st) {
  int ntiles = (MODE == Z_NEWTON || MODE == Z_FINAL) ? (a.nout > 3 ? 4 : 3) : 3;
  cudaError_t e = set_smem(k_zpass<N, MODE>, z_smem(4));
  if (e != cudaSuccess) return e;
  dim3 grid(YZCfg<N>::NBLK, N);
  k_zpass<N, MODE><<<grid, NT, z_smem(ntiles), st>>>(a);
  return cudaGetLastError();
}
}  // namespace

#define CAT2(a, b) a##b
#define CAT(a, b) CAT2(a, b)

cudaError_t CAT(mond_xpass_, MOND_N)(int mode, const passes::XArgs& a, cudaStream_t st) {
  switch (mode) {
    case X_RHO: return launch_x<X_RHO>(a, st);
    case X_NU_FIRST: return launch_xreg<X_NU_FIRST>(a, st);
    case X_NU: return launch_xreg<X_NU>(a, st);
    case X_MU: return launch_xreg<X_MU>(a, st);
    case X_INV: return launch_xreg<X_INV>(a, st);
    case X_FWD: return launch_xreg<X_FWD>(a, st);
    case X_NU_REAL: return launch_xreg<X_NU_REAL>(a, st);
    case X_DRHO: return launch_x<X_DRHO>(a, st);
    case X_DNU_FIRST: return launch_x<X_DNU_FIRST>(a, st);
    case X_DNU: return launch_x<X_DNU>(a, st);
    case X_DMU: return launch_x<X_DMU>(a, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t CAT(mond_ypass_, MOND_N)(int dir, const passes::YArgs& a, int ncomp, cudaStream_t st) {
  dim3 grid(YZCfg<N>::NBLK, N, ncomp);
  size_t sm = y_smem();
  if (dir < 0) {
    cudaError_t e = set_smem(k_ypass<N, -1>, sm);
    if (e != cudaSuccess) return e;
    k_ypass<N, -1><<<grid, NT, sm, st>>>(a);
  } else {
    cudaError_t e = set_smem(k_ypass<N, +1>, sm);
    if (e != cudaSuccess) return e;
    k_ypass<N, +1><<<grid, NT, sm, st>>>(a);
  }
  return cudaGetLastError();
}

namespace {
// The persistent grid: min(every CTA that fits, tiles, the caller's cap).
int capped(int grid, int ntiles, int cap) {
  int g = grid < ntiles ? grid : ntiles;
  return (cap > 0 && g > cap) ? cap : g;
}

template <typename K>
int pipe_grid(K kern, size_t sm, int nt = NT) {
  int dev = 0, sms = 1, per = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, nt, sm);
  return sms * (per > 0 ? per : 1);
}

template <int DIR>
cudaError_t launch_ypipe(const tma::TensorMap& map, const PipeYArgs& a, cudaStream_t st) {
  size_t sm = sizeof(float2) * (N + 2 * (size_t)N * PipeCfg<N>::PY);
  cudaError_t e = set_smem(k_ypass_pipe<N, DIR>, sm);
  if (e != cudaSuccess) return e;
  static int grid = 0;
  if (!grid) grid = pipe_grid(k_ypass_pipe<N, DIR>, sm);
  const int ntiles = PipeCfg<N>::NBLKY * N * a.ncomp;
  k_ypass_pipe<N, DIR><<<capped(grid, ntiles, a.max_ctas), NT, sm, st>>>(map, a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t CAT(mond_ypass_pipe_, MOND_N)(int dir, const tma::TensorMap& map, const passes::PipeYArgs& a,
                                          cudaStream_t st) {
  return dir < 0 ? launch_ypipe<-1>(map, a, st) : launch_ypipe<+1>(map, a, st);
}

namespace {
template <int KIND>
cudaError_t launch_yreg(const regpass::YRegArgs& a, int cap, cudaStream_t st) {
  using G = regpass::YGeo<N, KIND>;
  constexpr bool PAIR = KIND >= regpass::Y_FOLD;
  const size_t sm = sizeof(float2) * (N + (PAIR ? N / 2 + 2 * G::SLOTS : G::SLOTS));
  cudaError_t e = sm > 48 * 1024 ? set_smem(regpass::k_yreg<N, KIND>, sm) : cudaSuccess;
  if (e != cudaSuccess) return e;
  const int ntiles = G::TILES * (a.nplain + (PAIR ? 1 : 0));
  return launch_early(regpass::k_yreg<N, KIND>, capped(ntiles, ntiles, cap), G::T, sm, st, a, ntiles);
}

template <int MODE, bool FOLD, bool PHI>
cudaError_t launch_zreg(const regpass::ZRegArgs& a, int cap, cudaStream_t st) {
  using G = regpass::Geo<N>;
  const size_t sm = regpass::ZCfg<N, MODE, FOLD, PHI>::smem();
  cudaError_t e = sm > 48 * 1024 ? set_smem(regpass::k_zreg<N, MODE, FOLD, PHI>, sm) : cudaSuccess;
  if (e != cudaSuccess) return e;
  return launch_early(regpass::k_zreg<N, MODE, FOLD, PHI>, capped(G::TILES, G::TILES, cap), G::T, sm, st, a,
                      G::TILES);
}
}  // namespace

cudaError_t CAT(mond_yreg_, MOND_N)(int kind, const regpass::YRegArgs& a, int cap, cudaStream_t st) {
  switch (kind) {
    case regpass::Y_FWD: return launch_yreg<regpass::Y_FWD>(a, cap, st);
    case regpass::Y_INV: return launch_yreg<regpass::Y_INV>(a, cap, st);
    case regpass::Y_FOLD: return launch_yreg<regpass::Y_FOLD>(a, cap, st);
    case regpass::Y_CURL: return launch_yreg<regpass::Y_CURL>(a, cap, st);
    case regpass::Y_GRADN: return launch_yreg<regpass::Y_GRADN>(a, cap, st);
    case regpass::Y_GRAD: return launch_yreg<regpass::Y_GRAD>(a, cap, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t CAT(mond_zreg_, MOND_N)(int mode, bool fold, bool phi, const regpass::ZRegArgs& a, int cap,
                                    cudaStream_t st) {
  switch (mode) {
    case Z_NEWTON:
      if (fold) return phi ? launch_zreg<Z_NEWTON, true, true>(a, cap, st) : launch_zreg<Z_NEWTON, true, false>(a, cap, st);
      return phi ? launch_zreg<Z_NEWTON, false, true>(a, cap, st) : launch_zreg<Z_NEWTON, false, false>(a, cap, st);
    case Z_CURL:
      return fold ? launch_zreg<Z_CURL, true, false>(a, cap, st) : launch_zreg<Z_CURL, false, false>(a, cap, st);
    case Z_FINAL:
      if (fold) return phi ? launch_zreg<Z_FINAL, true, true>(a, cap, st) : launch_zreg<Z_FINAL, true, false>(a, cap, st);
      return phi ? launch_zreg<Z_FINAL, false, true>(a, cap, st) : launch_zreg<Z_FINAL, false, false>(a, cap, st);
    case Z_DIV: return launch_zreg<Z_DIV, false, false>(a, cap, st);
    case Z_SMOOTH: return launch_zreg<Z_SMOOTH, false, false>(a, cap, st);
  }
  return cudaErrorInvalidValue;
}

cudaError_t CAT(mond_zpass_, MOND_N)(int mode, const passes::ZArgs& a, cudaStream_t st) {
  switch (mode) {
    case Z_NEWTON: return launch_z<Z_NEWTON>(a, st);
    case Z_CURL: return launch_z<Z_CURL>(a, st);
    case Z_DIV: return launch_z<Z_DIV>(a, st);
    case Z_FINAL: return launch_z<Z_FINAL>(a, st);
    case Z_SMOOTH: return launch_z<Z_SMOOTH>(a, st);
  }
  return cudaErrorInvalidValue;
}
