// regpass.cuh -- the y- and z-passes of the field solve with their transforms
// in registers.
//
// A transform of length N = R0 R1 is two radix steps with one exchange between
// them. A thread first takes a butterfly of R0 values from global
// memory (rows j + r R1, 64-byte runs of 8 columns per row, copied into the
// slots that it then writes), then, after the exchange, one of R1 values, whose
// results are the frequencies j' + r R0. The
// inverse transform of a z-pass starts with the same R1 values, so that the
// spectral operator and the two radix steps around it happen on registers; its
// exchange runs back through the slots that each thread itself read, so that a
// pass over z has two barriers and touches a value in shared memory seven
// times, where the tiles staged by TMA took twelve and nine barriers.
//
// What bounds it: HBM at the larger sides (512^3 plain y-pass 6.2 TB/s, folded
// 5.3), registers and the latency of a tile at the smaller ones. Against the
// tiles staged by TMA (with a separate launch for the Nyquist tiles of a folded
// z-step), y- and z-passes of one K = 4 solve: 512^3 17.1 -> 14.6 ms, 256^3 1.58
// -> 1.57 ms, 192^3 1.12 -> 0.91 ms; the whole solve of 96^3, K = 3, 358 -> 288
// us.
#pragma once
#include <type_traits>

#include "passes.cuh"

namespace regpass {

using namespace passes;

// ---------------------------------------------------------------------------
// radix-R butterflies beyond those of fft.cuh
// ---------------------------------------------------------------------------
// cos and sin of 2 pi k / 24 and 2 pi k / 32, exact to FP32
__device__ __forceinline__ constexpr float cos24(int k) {
  constexpr float v[7] = {1.0f, 0.96592582628906829f, 0.86602540378443865f, 0.70710678118654752f, 0.5f,
                          0.25881904510252076f, 0.0f};
  k %= 24;
  if (k > 12) k = 24 - k;
  return k <= 6 ? v[k] : -v[12 - k];
}
__device__ __forceinline__ constexpr float sin24(int k) { return cos24(k + 18); }
__device__ __forceinline__ constexpr float cos32(int k) {
  constexpr float v[9] = {1.0f, 0.98078528040323044f, 0.92387953251128674f, 0.83146961230254524f,
                          0.70710678118654752f, 0.55557023301960222f, 0.38268343236508978f, 0.19509032201612827f, 0.0f};
  k %= 32;
  if (k > 16) k = 32 - k;
  return k <= 8 ? v[k] : -v[16 - k];
}
__device__ __forceinline__ constexpr float sin32(int k) { return cos32(k + 24); }

// radix 3 A (A = 2, 4, 8): three radix-A butterflies on the inputs 3 m + b, then
// radix 3 across them with W_{3A}^{b k}
template <int A, int DIR>
__device__ __forceinline__ void dft3x(float2* v) {
  float2 y[3][A];
#pragma unroll
  for (int b = 0; b < 3; b++) {
#pragma unroll
    for (int m = 0; m < A; m++) y[b][m] = v[3 * m + b];
    fftk::dftR<A, DIR>(y[b]);
  }
#pragma unroll
  for (int k = 0; k < A; k++) {
    constexpr int S = 24 / (3 * A);
    float2 t[3] = {y[0][k], cmul(y[1][k], make_float2(cos24(S * k), DIR * sin24(S * k))),
                   cmul(y[2][k], make_float2(cos24(2 * S * k), DIR * sin24(2 * S * k)))};
    fftk::dft3<DIR>(t);
    v[k] = t[0];
    v[k + A] = t[1];
    v[k + 2 * A] = t[2];
  }
}
template <int DIR>
__device__ __forceinline__ void dft32(float2* v) {
  float2 e[16], o[16];
#pragma unroll
  for (int i = 0; i < 16; i++) {
    e[i] = v[2 * i];
    o[i] = v[2 * i + 1];
  }
  fftk::dft16<DIR>(e);
  fftk::dft16<DIR>(o);
#pragma unroll
  for (int k = 0; k < 16; k++) {
    const float2 w = cmul(o[k], make_float2(cos32(k), DIR * sin32(k)));
    v[k] = cadd(e[k], w);
    v[k + 16] = csub(e[k], w);
  }
}
template <int R, int DIR>
__device__ __forceinline__ void dft(float2* v) {
  if constexpr (R == 6) dft3x<2, DIR>(v);
  else if constexpr (R == 12) dft3x<4, DIR>(v);
  else if constexpr (R == 24) dft3x<8, DIR>(v);
  else if constexpr (R == 32) dft32<DIR>(v);
  else fftk::dftR<R, DIR>(v);
}

// ---------------------------------------------------------------------------
// plan of a side: N = R0 R1 (R0 >= R1: the steps that hold several components
// are of radix R1), TC threads per sequence. Fewer threads with several
// butterflies each were slower (96: 288, 294, 353 us a solve with 12, 8, 4; 192:
// 1.93, 2.01, 2.11 ms a force evaluation with 16, 12, 8; 64: 293, 342 us with 8,
// 4; 128: 556, 579 us a step with 16, 8).
// ---------------------------------------------------------------------------
template <int N>
struct Plan;
#define MOND_RPLAN(NN, A, B, T)   \
  template <>                     \
  struct Plan<NN> {               \
    static constexpr int R0 = A, R1 = B, TC = T; \
  };
MOND_RPLAN(16, 4, 4, 4)
MOND_RPLAN(32, 8, 4, 4)
MOND_RPLAN(48, 8, 6, 8)
MOND_RPLAN(64, 8, 8, 8)
MOND_RPLAN(96, 12, 8, 12)
MOND_RPLAN(128, 16, 8, 16)
MOND_RPLAN(192, 16, 12, 16)
MOND_RPLAN(256, 16, 16, 16)
MOND_RPLAN(384, 24, 16, 24)
MOND_RPLAN(512, 32, 16, 16)
#undef MOND_RPLAN

// Sequences per tile: 8 columns of a row (two sectors; 16 columns measured 5 to
// 30% slower at 256, one CTA of twice the size per SM), or 8 rows of the column
// kx = N/2.
constexpr int PCOLS = 8;

// SWAP: the larger radix second (passes whose first step holds two values of
// each point and whose second holds one).
template <int N, bool SWAP = false>
struct Geo {
  using L = Plan<N>;
  static constexpr int P = PCOLS, R0 = SWAP ? L::R1 : L::R0, R1 = SWAP ? L::R0 : L::R1, TC = L::TC, T = P * TC, H = N / 2, SP = sp_of(N);
  // shared-memory slots: slot (j, r) of a sequence at (j (R0 + 1) + r) P + q, so
  // that both steps' accesses fall into distinct banks
  static constexpr int SLOTS = R1 * (R0 + 1) * P;
  static constexpr int COLS = H / P;         // tiles of 8 columns per row of the other axis
  static constexpr int TILES = COLS * N + N / P;  // and the tiles of the column kx = H
  static_assert(R0 * R1 == N && H % P == 0 && N % P == 0, "plan");
};

// CTAs per SM the passes are compiled for (registers: 65536 / (T ctas); 1: no
// limit). Without a limit the compiler takes 184 to 199 registers for the
// z-passes of 128 and 192, two CTAs per SM, and 144 to 150 for the pair
// y-passes, three. Per side, of a K = 4 solve:
//   192, z 3: divergence-free 57 -> 50 us, final 51 -> 43 (4: no gain);
//        pair y 4: fold 39 -> 34 us, unfold 34 -> 31 (5: no gain); plain y 7:
//        a force step 1701 -> 1695 us;
//   128, a step of two particles: z 3: 543 -> 534 us, and pair y 4: 529,
//        and z 4: 515 (5: 524);
//   256, z 3 / 4: divergence-free 116 / 126 us (spills), folded final 104 /
//        121; pair y 4 / 5: 73 / 71 and 68 / 70;
//   384 (T = 192: one CTA per SM without a limit, both kinds), a K = 4 solve:
//        13.1 ms; z 2: 12.0, and pair y 2: 10.9, 3: 10.6, and plain y 4: 10.2
//        (16 threads a sequence with limits to match: 10.5);
//   512, pair y 3 instead of 2: a K = 4 solve 23.7 -> 23.4 ms (z 3, pair y 4,
//        plain y 5: no gain);
//   64, 96: no difference.
constexpr int zctas(int n) { return n == 128 ? 4 : n == 192 || n == 256 ? 3 : n == 384 ? 2 : 1; }
constexpr int yctas(int n, bool pair) {
  if (pair) return n >= 384 ? 3 : n >= 128 ? 4 : 1;
  return n == 192 ? 7 : n == 384 ? 4 : 1;
}

// The exchange slot of butterfly j, value r, of this thread's sequence.
template <class G>
__device__ __forceinline__ int slot(int j, int r) {
  return (j * (G::R0 + 1) + r) * G::P;
}

// tile -> this thread's column and its index on the other (untransformed) axis
template <int N>
__device__ __forceinline__ bool tile_of(int t, int q, int& col, int& row) {
  using G = Geo<N>;
  if (t < G::COLS * N) {
    col = (t % G::COLS) * G::P + q;
    row = t / G::COLS;
    return false;
  }
  col = G::H;
  row = (t - G::COLS * N) * G::P + q;
  return true;
}

// Copies n bytes (a multiple of 16) of a table to shared memory, asynchronously
// (complete after async_wait_all and a barrier). The tables are read from
// there: the streamed data would push them out of the small L1 that the
// exchange leaves.
__device__ __forceinline__ void table_in(void* dst, const void* src, int n, int tid, int nt) {
  for (int i = 16 * tid; i < n; i += 16 * nt)
    tma::async_copy16(static_cast<char*>(dst) + i, static_cast<const char*>(src) + i);
}

// Starts the copies of a tile's values into the slots of their first step:
// position j + r R1 of the sequence to slot (j, r); complete after
// async_wait_all and __syncwarp (two lanes of a warp copy 16 bytes, two
// columns, for each other; the column kx = H goes value by value). g: this
// lane's sequence, rs: between its positions, sm: its slots. Loads to registers
// would be held in what the exchange leaves of the L1 while in flight: 256^3
// z-passes took longer with four CTAs per SM than with three.
template <class G>
__device__ __forceinline__ void fetch(float2* sm, const float2* g, int64_t rs, bool colH, int q, int tt) {
  const int odd = q & 1;
  for (int j = tt; j < G::R1; j += G::TC) {
    if (!colH) {
#pragma unroll
      for (int i = 0; i < G::R0 / 2; i++) {
        const int r = 2 * i + odd;
        tma::async_copy16(sm - odd + slot<G>(j, r), g - odd + (j + r * G::R1) * rs);
      }
    } else {
#pragma unroll
      for (int r = 0; r < G::R0; r++) tma::async_copy8(sm + slot<G>(j, r), g + (j + r * G::R1) * rs);
    }
  }
}
__device__ __forceinline__ void fetched() {
  tma::async_wait_all();
  __syncwarp();
}

// First radix step: butterfly j, from and to its slots.
template <class G, int DIR>
__device__ __forceinline__ void step0(float2* v, float2* sm, int j) {
  dft<G::R0, DIR>(v);
#pragma unroll
  for (int r = 0; r < G::R0; r++) sm[slot<G>(j, r)] = v[r];
}
template <class G, int DIR>
__device__ __forceinline__ void step0(float2* sm, int j) {
  float2 v[G::R0];
#pragma unroll
  for (int r = 0; r < G::R0; r++) v[r] = sm[slot<G>(j, r)];
  step0<G, DIR>(v, sm, j);
}
// Second radix step: butterfly j from the slots; v[r] is position j + r R0.
template <class G, int DIR>
__device__ __forceinline__ void step1(float2* v, const float2* sm, int j, const float2* tw) {
  constexpr int R1 = G::R1;
#pragma unroll
  for (int r = 0; r < R1; r++) v[r] = sm[slot<G>(r, j)];
#pragma unroll
  for (int r = 1; r < R1; r++) v[r] = cmul(v[r], twid<DIR>(tw[r * j]));
  dft<R1, DIR>(v);
}
// First step of the inverse, in place of step1's slots.
template <class G>
__device__ __forceinline__ void istep0(float2* v, float2* sm, int j) {
  dft<G::R1, +1>(v);
#pragma unroll
  for (int r = 0; r < G::R1; r++) sm[slot<G>(r, j)] = v[r];
}
// Second step of the inverse from step0's slots; v[r] is position j + r R1.
template <class G>
__device__ __forceinline__ void istep1(float2* v, const float2* sm, int j, const float2* tw) {
  constexpr int R0 = G::R0;
#pragma unroll
  for (int r = 0; r < R0; r++) v[r] = sm[slot<G>(j, r)];
#pragma unroll
  for (int r = 1; r < R0; r++) v[r] = cmul(v[r], tw[r * j]);
  dft<R0, +1>(v);
}

// ---------------------------------------------------------------------------
// y-passes
//
// Folded: away from the Nyquist planes the curl-free projection k (k.g) A is the
// gradient of one scalar, and so are the final and Newton operators. The y-pass
// before such a z-pass folds the x and y components into s = kx gx^ + ky gy^
// (component 0; component 2 keeps gz^), the z-pass takes the two and returns the
// scalar u and the z component, and the y-pass after it unfolds u into kx u and
// ky u ahead of its transform. On the column kx = N/2 and the row ky = N/2 the
// Nyquist rule of the projection splits the axes into two sets, so that gx^ and
// gy^ stay apart there (components 0 and 1) and the z-pass works on three
// components; for Newton, kappa vanishes there and everything is folded.
// ---------------------------------------------------------------------------
enum YKind {
  Y_FWD = 0,       // plain, components c0 .. c0 + nplain - 1
  Y_INV = 1,
  Y_FOLD = 2,      // forward: s = kx gx^ + ky gy^ into component 0, then the plain components
  Y_CURL = 3,      // inverse after the curl-free z-pass: kx u, ky u (kt = k)
  Y_GRADN = 4,     // inverse after the final z-pass: kappa_x u, kappa_y u (kt = kappa)
  Y_GRAD = 5       // inverse after the Newton z-pass: as Y_GRADN, nothing apart on the Nyquist planes
};

struct YRegArgs {
  float2* spec;
  int64_t pstride;   // complex elements between components
  int c0, nplain;    // components transformed as they are
  const float2* tw;
  const float* kt;   // per index: k (fold, curl) or kappa (gradients)
};

// The unfolding passes hold two values of a point in their first step.
template <int N, int KIND>
using YGeo = Geo<N, (KIND > Y_FOLD)>;

// Where the folded passes keep components apart (gx^ in component 0, gy^ in
// component 1): the column kx = N/2, and the row ky = N/2.
template <int N, int KIND>
__global__ void __launch_bounds__(YGeo<N, KIND>::T, yctas(N, KIND >= Y_FOLD)) k_yreg(YRegArgs a, int ntiles) {
  using G = YGeo<N, KIND>;
  constexpr int R0 = G::R0, R1 = G::R1, H = G::H, SP = G::SP;
  constexpr bool PAIR = KIND >= Y_FOLD;
  constexpr int DIR = (KIND == Y_FWD || KIND == Y_FOLD) ? -1 : +1;
  extern __shared__ __align__(16) float2 rsm[];
  const int q = threadIdx.x % G::P, tt = threadIdx.x / G::P;
  // tables: twiddles, then (pair) kt
  float2* const tw = rsm;
  float* const kt = reinterpret_cast<float*>(rsm + N);
  float2* const sm = rsm + N + (PAIR ? N / 2 : 0) + q;
  float2* const sm1 = sm + G::SLOTS;
  table_in(tw, a.tw, 8 * N, threadIdx.x, G::T);
  if (PAIR) table_in(kt, a.kt, 4 * N, threadIdx.x, G::T);
  kernel_wait();
  bool first = true;
  for (int t0 = blockIdx.x; t0 < ntiles; t0 += gridDim.x) {
    if (!first) __syncthreads();
    first = false;
    // the pair's tiles first, then the plain components'
    const int grp = t0 / G::TILES, t = t0 - grp * G::TILES;
    const bool pair = PAIR && grp == 0;
    int col, z;
    const bool colH = tile_of<N>(t, q, col, z);
    const int64_t at = (int64_t)z * N * SP + col;
    if (!pair) {
      float2* const g = a.spec + (a.c0 + grp - (PAIR ? 1 : 0)) * a.pstride + at;
      fetch<G>(sm, g, SP, colH, q, tt);
      fetched();
      for (int j = tt; j < R1; j += G::TC) step0<G, DIR>(sm, j);
      __syncthreads();
      for (int j = tt; j < R0; j += G::TC) {
        float2 v[R1];
        step1<G, DIR>(v, sm, j, tw);
#pragma unroll
        for (int r = 0; r < R1; r++) g[(j + r * R0) * SP] = v[r];
      }
      continue;
    }
    if constexpr (PAIR) {
      float2* const g0 = a.spec + at;
      float2* const g1 = g0 + a.pstride;
      const float kx = __ldg(a.kt + col);
      if constexpr (KIND == Y_FOLD) {
        fetch<G>(sm, g0, SP, colH, q, tt);
        fetch<G>(sm1, g1, SP, colH, q, tt);
        fetched();
        for (int j = tt; j < R1; j += G::TC) {
          step0<G, DIR>(sm, j);
          step0<G, DIR>(sm1, j);
        }
        __syncthreads();
        for (int j = tt; j < R0; j += G::TC) {
          float2 x[R1], y[R1];
          step1<G, DIR>(x, sm, j, tw);
          step1<G, DIR>(y, sm1, j, tw);
#pragma unroll
          for (int r = 0; r < R1; r++) {
            const int row = j + r * R0;
            if (colH || row == H) {
              g0[row * SP] = x[r];
              g1[row * SP] = y[r];
            } else {
              g0[row * SP] = cadd(cscale(x[r], kx), cscale(y[r], kt[row]));
            }
          }
        }
      } else {
        fetch<G>(sm, g0, SP, colH, q, tt);
        if (KIND != Y_GRAD && colH) fetch<G>(sm1, g1, SP, colH, q, tt);
        fetched();
        __syncthreads();  // the table kt
        for (int j = tt; j < R1; j += G::TC) {
          float2 v[R0];
          if (KIND != Y_GRAD && colH) {
            step0<G, DIR>(sm, j);
            step0<G, DIR>(sm1, j);
            continue;
          }
#pragma unroll
          for (int r = 0; r < R0; r++) {
            const int row = j + r * R1;
            v[r] = cscale(sm[slot<G>(j, r)], kt[row]);
            if (KIND != Y_GRAD && row == H) v[r] = __ldcg(g1 + row * SP);
          }
          step0<G, DIR>(v, sm1, j);
#pragma unroll
          for (int r = 0; r < R0; r++) {
            v[r] = sm[slot<G>(j, r)];
            if (KIND == Y_GRAD || j + r * R1 != H) v[r] = cscale(v[r], kx);
          }
          step0<G, DIR>(v, sm, j);
        }
        __syncthreads();
        for (int j = tt; j < R0; j += G::TC) {
          float2 v[R1];
          step1<G, DIR>(v, sm, j, tw);
#pragma unroll
          for (int r = 0; r < R1; r++) g0[(j + r * R0) * SP] = v[r];
          step1<G, DIR>(v, sm1, j, tw);
#pragma unroll
          for (int r = 0; r < R1; r++) g1[(j + r * R0) * SP] = v[r];
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// z-passes
// ---------------------------------------------------------------------------
struct ZRegArgs {
  const float2* in;
  float2* out;
  float2* scal;      // component 3 of the final spectra: the kept potential of the mean, or the potential
  int64_t pstride;
  int mean;          // 1: Z_CURL writes its potential to scal, 2: Z_FINAL takes the mean with scal
  const float* kv;
  const float* kp;
  const float2* tw;
  const float* khat;
  float norm;
  float coef;
};

// The spectral operator at one point on the components of g (in place); sc: the
// point's scalar, in (mean of two iterations) and out (potential). n*: the
// axis is on its Nyquist plane.
template <int MODE>
__device__ __forceinline__ void zop3(const ZRegArgs& a, float kx, float ky, float kz, float kpx, float kpy, float kpz,
                                     bool nx, bool ny, bool nz, float fk, float2* g, float2& sc) {
  const float kk = kx * kx + ky * ky + kz * kz;
  const float A = kk > 0.f ? __frcp_rn(kk) : 0.f;  // correctly rounded, as 1.0f / kk
  const float k3[3] = {kx, ky, kz};
  const bool n3[3] = {nx, ny, nz};
  if constexpr (MODE == Z_NEWTON) {
    const float f = a.coef * A * a.norm;  // 4 pi G A / N^3
    const float2 r = g[0], ir = cmul_i<1>(r);
    g[0] = cscale(ir, f * kpx);
    g[1] = cscale(ir, f * kpy);
    g[2] = cscale(ir, f * kpz);
    sc = cscale(r, -f);  // phi_N^ = -4 pi G A rho^
  } else if constexpr (MODE == Z_SMOOTH) {
    const float f = fk * a.norm;
    for (int c = 0; c < 3; c++) g[c] = cscale(g[c], f);
  } else if constexpr (MODE == Z_FINAL) {
    // phi^ = i A sum_b k'_b g_b (k'_b = 0 on b's Nyquist plane); a^ = -i kappa phi^
    float2 S = make_float2(0.f, 0.f);
    for (int b = 0; b < 3; b++)
      if (!n3[b]) S = cadd(S, cscale(g[b], k3[b]));
    float2 aS = cscale(S, A * a.norm);
    if (a.mean == 2) aS = cscale(cadd(aS, sc), 0.5f);  // the midpoint of the last two iterations
    const float2 aK = cscale(aS, fk);  // times the smoothing spectrum when the mesh is to hold the node-smoothed field
    g[0] = cscale(aK, kpx);
    g[1] = cscale(aK, kpy);
    g[2] = cscale(aK, kpz);
    sc = cmul_i<1>(aS);
  } else if (!(nx || ny || nz)) {
    // away from the Nyquist planes: P g = k (k.g) A, from one dot product
    const float2 S = cadd(cadd(cscale(g[0], kx), cscale(g[1], ky)), cscale(g[2], kz));
    const float2 SA = cscale(S, A);
    sc = cscale(SA, a.norm);  // the potential this step implies, as Z_FINAL forms it
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const float2 t = cscale(SA, k3[c]);
      g[c] = cscale((MODE == Z_DIV) ? csub(g[c], t) : t, a.norm);
    }
  } else {
    float2 S = make_float2(0.f, 0.f);
    for (int b = 0; b < 3; b++)
      if (!n3[b]) S = cadd(S, cscale(g[b], k3[b]));
    sc = cscale(S, A * a.norm);
    // P_ab = k_a k_b A, off-diagonal terms dropped when exactly one of a, b is on its Nyquist plane
    float2 o[3];
    for (int c = 0; c < 3; c++) {
      float2 t = make_float2(0.f, 0.f);
      for (int b = 0; b < 3; b++)
        if (c == b || n3[c] == n3[b]) t = cadd(t, cscale(g[b], k3[c] * k3[b] * A));
      o[c] = cscale((MODE == Z_DIV) ? csub(g[c], t) : t, a.norm);
    }
    for (int c = 0; c < 3; c++) g[c] = o[c];
  }
}

// FOLD: the folded pair (components 0 and 2) where nothing is on a Nyquist
// plane of x or y, three components where something is (none for Newton).
// PHI: the potential too (its inverse z transform, component 3).
template <int N, int MODE, bool FOLD, bool PHI>
struct ZCfg {
  static constexpr bool FAST = FOLD || MODE == Z_DIV;            // the operator in registers away from the Nyquist planes
  static constexpr bool SLOW = !(FOLD && MODE == Z_NEWTON);      // has tiles whose operator runs through the slots
  static constexpr int REGIONS = (SLOW ? 3 : 2) + (PHI ? 1 : 0);
  static constexpr size_t smem() { return sizeof(float2) * (2 * N + REGIONS * Geo<N>::SLOTS); }
};

template <int N, int MODE, bool FOLD, bool PHI>
__global__ void __launch_bounds__(Geo<N>::T, zctas(N)) k_zreg(ZRegArgs a, int ntiles) {
  using G = Geo<N>;
  using C = ZCfg<N, MODE, FOLD, PHI>;
  constexpr int R0 = G::R0, R1 = G::R1, H = G::H, SP = G::SP, SL = G::SLOTS;
  constexpr int64_t RS = (int64_t)N * SP;  // between z rows
  extern __shared__ __align__(16) float2 rsm[];
  const int q = threadIdx.x % G::P, tt = threadIdx.x / G::P;
  // tables: twiddles, k, kappa; then component c at sm + c SL, the potential last
  float2* const tw = rsm;
  float* const kv = reinterpret_cast<float*>(rsm + N);
  float* const kp = kv + N;
  float2* const sm = rsm + 2 * N + q;
  table_in(tw, a.tw, 8 * N, threadIdx.x, G::T);
  table_in(kv, a.kv, 4 * N, threadIdx.x, G::T);
  table_in(kp, a.kp, 4 * N, threadIdx.x, G::T);
  kernel_wait();
  const bool mean_in = MODE == Z_FINAL && a.mean == 2, mean_out = MODE == Z_CURL && a.mean == 1;
  const bool use_khat = MODE == Z_SMOOTH || (MODE == Z_FINAL && a.khat);
  bool first = true;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    if (!first) __syncthreads();
    first = false;
    int col, y;
    const bool colH = tile_of<N>(t, q, col, y);
    const int64_t at = (int64_t)y * SP + col;
    const float kx = __ldg(a.kv + col), ky = __ldg(a.kv + y);
    const bool fast = C::FAST && (!C::SLOW || !(colH || y == H));  // the same for all threads
    auto scal_at = [&](int row) { return a.scal + row * RS + at; };
    auto fk_at = [&](int row) {
      return use_khat ? __ldg(a.khat + ((int64_t)row * N + y) * (N / 2 + 1) + col) : 1.0f;
    };
    auto inv_k2 = [&](float kz) {
      const float kk = kx * kx + ky * ky + kz * kz;
      return kk > 0.f ? __frcp_rn(kk) : 0.f;  // correctly rounded, as 1.0f / kk
    };
    auto store = [&](float2* g, const float2* s, int j) {
      float2 v[R0];
      istep1<G>(v, s, j, tw);
#pragma unroll
      for (int r = 0; r < R0; r++) g[(j + r * R1) * RS] = v[r];
    };
    if (fast) {
      // regions: s, gz (folded; out u and the z component) or the three components
      constexpr int NIN = MODE == Z_NEWTON ? 1 : (FOLD ? 2 : 3), NOUT = FOLD ? 2 : 3;
#pragma unroll
      for (int c = 0; c < NIN; c++) fetch<G>(sm + c * SL, a.in + (FOLD && c ? 2 : c) * a.pstride + at, RS, colH, q, tt);
      fetched();
      for (int j = tt; j < R1; j += G::TC)
#pragma unroll
        for (int c = 0; c < NIN; c++) step0<G, -1>(sm + c * SL, j);
      __syncthreads();
      for (int j = tt; j < R0; j += G::TC) {
        float2 v[R1], S[R1];
        if constexpr (MODE == Z_DIV) {
          // S = k.g; the x and y components go back to their slots meanwhile
          step1<G, -1>(v, sm, j, tw);
#pragma unroll
          for (int r = 0; r < R1; r++) {
            S[r] = cscale(v[r], kx);
            sm[slot<G>(r, j)] = v[r];
          }
          step1<G, -1>(v, sm + SL, j, tw);
#pragma unroll
          for (int r = 0; r < R1; r++) {
            S[r] = cadd(S[r], cscale(v[r], ky));
            sm[SL + slot<G>(r, j)] = v[r];
          }
          step1<G, -1>(v, sm + 2 * SL, j, tw);
#pragma unroll
          for (int r = 0; r < R1; r++) {
            const int row = j + r * R0;
            const float kz = kv[row], A = inv_k2(kz);
            // kz on its Nyquist plane: z is a set of its own
            const float2 tz = row == H ? cscale(v[r], kz) : cadd(S[r], cscale(v[r], kz));
            v[r] = cscale(csub(v[r], cscale(tz, kz * A)), a.norm);
            S[r] = cscale(row == H ? S[r] : tz, A);
          }
          istep0<G>(v, sm + 2 * SL, j);
#pragma unroll
          for (int c = 0; c < 2; c++) {
            const float kc = c ? ky : kx;
#pragma unroll
            for (int r = 0; r < R1; r++) v[r] = cscale(csub(sm[c * SL + slot<G>(r, j)], cscale(S[r], kc)), a.norm);
            istep0<G>(v, sm + c * SL, j);
          }
        } else {
          // u, then the z component from it (kz u, kappa_z u)
          float2 sc[MODE == Z_FINAL ? R1 : 1];
          if constexpr (MODE == Z_FINAL) {
            if (mean_in) {
#pragma unroll
              for (int r = 0; r < R1; r++) sc[r] = __ldcg(scal_at(j + r * R0));
            }
          }
          step1<G, -1>(S, sm, j, tw);
          if constexpr (MODE != Z_NEWTON) step1<G, -1>(v, sm + SL, j, tw);
#pragma unroll
          for (int r = 0; r < R1; r++) {
            const int row = j + r * R0;
            const float kz = kv[row], A = inv_k2(kz);
            if constexpr (MODE == Z_NEWTON) {
              const float f = a.coef * A * a.norm;  // 4 pi G A / N^3
              if constexpr (PHI) v[r] = cscale(S[r], -f);  // phi_N^ = -4 pi G A rho^
              S[r] = cscale(cmul_i<1>(S[r]), f);
            } else if constexpr (MODE == Z_CURL) {
              const float2 u = row == H ? S[r] : cadd(S[r], cscale(v[r], kz));
              S[r] = cscale(cscale(u, A), a.norm);
              v[r] = row == H ? cscale(v[r], kz * kz * A * a.norm) : cscale(S[r], kz);
              if (mean_out) *scal_at(row) = S[r];  // the potential this step implies, as Z_FINAL forms it
            } else {
              // phi^ = i A sum_b k'_b g_b (k'_z = 0 on its Nyquist plane), a^ = -i kappa phi^
              float2 u = row == H ? S[r] : cadd(S[r], cscale(v[r], kz));
              u = cscale(u, A * a.norm);
              if (mean_in) u = cscale(cadd(u, sc[r]), 0.5f);  // the midpoint of the last two iterations
              if constexpr (PHI) v[r] = cmul_i<1>(u);
              S[r] = cscale(u, fk_at(row));
            }
          }
          if constexpr (PHI) istep0<G>(v, sm + (C::REGIONS - 1) * SL, j);
          if constexpr (MODE != Z_CURL) {
#pragma unroll
            for (int r = 0; r < R1; r++) v[r] = cscale(S[r], kp[j + r * R0]);
          }
          istep0<G>(v, sm + SL, j);
          istep0<G>(S, sm, j);
        }
      }
      __syncthreads();
      for (int j = tt; j < R1; j += G::TC) {
#pragma unroll
        for (int c = 0; c < NOUT; c++) store(a.out + (FOLD && c ? 2 : c) * a.pstride + at, sm + c * SL, j);
        if constexpr (PHI) store(a.scal + at, sm + (C::REGIONS - 1) * SL, j);
      }
    } else if constexpr (C::SLOW) {
      // three components, the operator through the slots: a thread reads and
      // writes its own slots only between the barriers
      constexpr int NIN = MODE == Z_NEWTON ? 1 : 3;
      const float kpx = __ldg(a.kp + col), kpy = __ldg(a.kp + y);
      for (int c = 0; c < NIN; c++) fetch<G>(sm + c * SL, a.in + c * a.pstride + at, RS, colH, q, tt);
      fetched();
      for (int j = tt; j < R1; j += G::TC)
        for (int c = 0; c < NIN; c++) step0<G, -1>(sm + c * SL, j);
      __syncthreads();
      for (int j = tt; j < R0; j += G::TC) {
        for (int c = 0; c < NIN; c++) {
          float2 v[R1];
          step1<G, -1>(v, sm + c * SL, j, tw);
#pragma unroll
          for (int r = 0; r < R1; r++) sm[c * SL + slot<G>(r, j)] = v[r];
        }
        for (int r = 0; r < R1; r++) {
          const int row = j + r * R0;
          float2* s = sm + slot<G>(r, j);
          float2 g[3] = {s[0], s[SL], s[2 * SL]}, sc = make_float2(0.f, 0.f);
          if (mean_in) sc = *scal_at(row);
          zop3<MODE>(a, kx, ky, kv[row], kpx, kpy, kp[row], colH, y == H, row == H, fk_at(row), g,
                     sc);
          if (mean_out) *scal_at(row) = sc;
          for (int c = 0; c < 3; c++) s[c * SL] = g[c];
          if (PHI) s[(C::REGIONS - 1) * SL] = sc;
        }
        for (int c = 0; c < C::REGIONS; c++) {
          float2 v[R1];
#pragma unroll
          for (int r = 0; r < R1; r++) v[r] = sm[c * SL + slot<G>(r, j)];
          istep0<G>(v, sm + c * SL, j);
        }
      }
      __syncthreads();
      for (int j = tt; j < R1; j += G::TC)
        for (int c = 0; c < C::REGIONS; c++)
          store(c == 3 ? a.scal + at : a.out + c * a.pstride + at, sm + c * SL, j);
    }
  }
}

}  // namespace regpass
