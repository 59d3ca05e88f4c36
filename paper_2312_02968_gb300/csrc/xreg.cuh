// xreg.cuh -- the x-passes of the field solve with their transforms in
// registers: C2R, the pointwise step of the iteration, R2C, on contiguous lines.
//
// A line of N reals is a complex transform of length H = N/2 = A0 A1 plus the
// pre- and post-processing of a real one. TL lanes of a warp own a line, so
// that a warp needs no barrier but its own. The spectrum comes in by 16-byte
// asynchronous copies; a lane takes the butterflies j and A1 - j (A0 values
// each) together, because the real transform couples position k with H - k,
// which lies in them; after one exchange through shared memory it has A1
// positions of real space per component, where the pointwise step runs, and
// the way back mirrors the way in, up to the direct store of the spectrum.
//
// What bounds it: HBM (the fields are larger than L2 from 192^3 on), at 0.74 of
// the copy rate; the earlier kernel was bound by shared memory, 16 accesses a
// value and a barrier per step (89% of its data pipe at 256), where this one
// makes nine. A launch at 256^3 (deep MOND): nu 0.166 -> 0.134 ms, mu 0.158 ->
// 0.119, inverse 0.094 -> 0.074; at 512^3 nu 1.61 -> 1.08, mu 1.53 -> 1.03.
#pragma once
#include "regpass.cuh"

namespace xreg {

using namespace passes;
using regpass::dft;

// plan of a side: H = A0 A1, TL lanes per line
template <int N>
struct Plan;
#define MOND_XPLAN(NN, A, B, T)   \
  template <>                     \
  struct Plan<NN> {               \
    static constexpr int A0 = A, A1 = B, TL = T; \
  };
MOND_XPLAN(16, 2, 4, 2)
MOND_XPLAN(32, 4, 4, 4)
MOND_XPLAN(48, 4, 6, 4)
MOND_XPLAN(64, 4, 8, 4)
MOND_XPLAN(96, 6, 8, 8)
MOND_XPLAN(128, 8, 8, 8)
MOND_XPLAN(192, 8, 12, 8)
MOND_XPLAN(256, 8, 16, 8)
MOND_XPLAN(384, 12, 16, 8)
MOND_XPLAN(512, 16, 16, 16)
#undef MOND_XPLAN

constexpr int WARPS = 4;  // per CTA; each on lines of its own

template <int N>
struct Geo {
  static constexpr int A0 = Plan<N>::A0, A1 = Plan<N>::A1, TL = Plan<N>::TL, H = N / 2, SP = sp_of(N);
  static constexpr int LW = 32 / TL;    // lines per warp
  static constexpr int HALF = A1 / 2;   // butterfly pairs (j, A1 - j)
  // value k of a line at (k / A1) G + k mod A1: groups padded so that 16-byte
  // reads of whole groups by neighbouring lanes fall into distinct banks
  static constexpr int G = A1 + (A1 == 6 ? 4 : 2);
  // line pitch: room for k = H and its pad column; lines of a half warp offset
  // so that the 8-byte accesses of their lanes do not collide
  static constexpr int WANT = TL >= 16 ? 8 : TL % 16;  // pitch mod 16 values
  static constexpr int PITCH = (A0 * G + 2 - WANT + 15) / 16 * 16 + WANT;
  static constexpr int REGION = LW * PITCH;  // one component of a warp's lines
  static constexpr int LINES = LW * WARPS;   // per CTA
  static_assert(A0 * A1 == H && A0 % 2 == 0 && A1 % 2 == 0 && (N * N) % LINES == 0 && PITCH >= A0 * G + 2, "plan");
};

// Whether a mode has an inverse (C2R) and a forward (R2C) part, and the
// components held together.
constexpr bool has_inv(int m) { return m == X_NU_FIRST || m == X_NU || m == X_MU || m == X_INV; }
constexpr bool has_fwd(int m) { return m != X_INV; }
constexpr int ncomp_of(int m) { return (m == X_INV || m == X_FWD) ? 1 : 3; }
template <int N, int MODE>
constexpr size_t smem_bytes() {
  return sizeof(float2) * (N + (size_t)WARPS * ncomp_of(MODE) * Geo<N>::REGION);
}

// CTAs per SM the three-component modes are compiled for. 192: 4 (128 instead of
// 136 registers) nu 95 -> 81 us; 128: 5, eight systems side by side 1% less (6:
// 1% more); 256: what shared memory admits; 64, 96: more made no difference.
constexpr int xctas(int n) { return n == 192 ? 4 : n == 128 ? 5 : 3; }

// 16-byte asynchronous copy whose source lines leave L2 first (read once).
__device__ __forceinline__ void copy16_stream(void* dst, const void* src, uint64_t policy) {
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(tma::smem_addr(dst)), "l"(src),
               "l"(policy)
               : "memory");
}

// Y[k] of the half-length inverse transform from X[k] = a and X[H - k] = b, w =
// e^{2 pi i k/N}: (a + conj b) + i w (a - conj b).
__device__ __forceinline__ float2 pre1(float2 a, float2 b, float2 w) {
  const float2 bc = cconj(b);
  return cadd(cadd(a, bc), cmul_i<1>(cmul(w, csub(a, bc))));
}
// X[k] from Z[k] = a and Z[H - k] = b: E - i conj(w) D, E, D = (a +- conj b)/2.
__device__ __forceinline__ float2 post1(float2 a, float2 b, float2 w) {
  const float2 bc = cconj(b);
  const float2 e = cscale(cadd(a, bc), 0.5f), d = cscale(csub(a, bc), 0.5f);
  return csub(e, cmul_i<1>(cmul(cconj(w), d)));
}

// First step of the inverse: butterflies j0 = m and j1 = A1 - m (m = 0: 0 and
// A1/2) of a line's half spectrum, pre-processed, transformed over their A0
// values and put back into the same places.
template <int N>
__device__ __forceinline__ void inv_pair(float2* s, int m, const float2* tw) {
  using X = Geo<N>;
  constexpr int A0 = X::A0, A1 = X::A1, G = X::G;
  const int j0 = m, j1 = m ? A1 - m : A1 / 2;
  const bool z = m == 0;
  float2 a[A0], b[A0];
#pragma unroll
  for (int r = 0; r < A0; r++) {
    a[r] = s[j0 + G * r];
    b[r] = s[j1 + G * r];
  }
  float2 ya[A0], yb[A0];
#pragma unroll
  for (int r = 0; r < A0; r++) {
    // position H - k: of a[r] in the other butterfly, at A0 - 1 - r; m = 0: both are their own partners
    const float2 own = r ? a[A0 - r] : s[A0 * G];
    float2 pa = z ? own : b[A0 - 1 - r];
    const float2 pb = z ? b[A0 - 1 - r] : a[A0 - 1 - r];
    float2 x = a[r];
    if (r == 0) {  // the imaginary parts of X[0] and X[H] are dropped (real part of the inverse)
      x.y = z ? 0.f : x.y;
      pa.y = z ? 0.f : pa.y;
    }
    ya[r] = pre1(x, pa, tw[j0 + A1 * r]);
    yb[r] = pre1(b[r], pb, tw[j1 + A1 * r]);
  }
  dft<A0, +1>(ya);
  dft<A0, +1>(yb);
#pragma unroll
  for (int r = 0; r < A0; r++) {
    s[j0 + G * r] = ya[r];
    s[j1 + G * r] = yb[r];
  }
}

// Last step of the forward transform: butterflies j0 and j1, post-processed and
// stored to the spectral row g.
template <int N>
__device__ __forceinline__ void fwd_pair(const float2* s, int m, const float2* tw, float2* g) {
  using X = Geo<N>;
  constexpr int A0 = X::A0, A1 = X::A1, G = X::G, H = X::H;
  const int j0 = m, j1 = m ? A1 - m : A1 / 2;
  const bool z = m == 0;
  float2 a[A0], b[A0];
#pragma unroll
  for (int r = 0; r < A0; r++) {
    a[r] = s[j0 + G * r];
    b[r] = s[j1 + G * r];
  }
  dft<A0, -1>(a);
  dft<A0, -1>(b);
#pragma unroll
  for (int r = 0; r < A0; r++) {
    const float2 own = a[r ? A0 - r : 0];
    const float2 pa = z ? own : b[A0 - 1 - r];
    const float2 pb = z ? b[A0 - 1 - r] : a[A0 - 1 - r];
    float2 xa = post1(a[r], pa, tw[j0 + A1 * r]);
    if (r == 0 && z) {
      // k = 0 and k = H from Z[0]; the pad columns past H are left as they are
      // (read with their neighbours by wide copies, used by nothing)
      xa = make_float2(a[0].x + a[0].y, 0.f);
      g[H] = make_float2(a[0].x - a[0].y, 0.f);
    }
    __stcs(g + j0 + A1 * r, xa);
    __stcs(g + j1 + A1 * r, post1(b[r], pb, tw[j1 + A1 * r]));
  }
}

// Second step of the inverse of butterfly p: v[s] is position p + A0 s.
template <int N>
__device__ __forceinline__ void inv_mid(float2* v, const float2* s, int p, const float2* tw) {
  constexpr int A1 = Geo<N>::A1;
  const float4* q = reinterpret_cast<const float4*>(s + p * Geo<N>::G);
#pragma unroll
  for (int j = 0; j < A1 / 2; j++) {
    const float4 t = q[j];
    v[2 * j] = make_float2(t.x, t.y);
    v[2 * j + 1] = make_float2(t.z, t.w);
  }
#pragma unroll
  for (int j = 1; j < A1; j++) v[j] = cmul(v[j], tw[2 * j * p]);
  dft<A1, +1>(v);
}
// First step of the forward transform, to the same places.
template <int N>
__device__ __forceinline__ void fwd_mid(float2* v, float2* s, int p, const float2* tw) {
  constexpr int A1 = Geo<N>::A1;
  dft<A1, -1>(v);
#pragma unroll
  for (int j = 1; j < A1; j++) v[j] = cmul(v[j], cconj(tw[2 * j * p]));
  float4* q = reinterpret_cast<float4*>(s + p * Geo<N>::G);
#pragma unroll
  for (int j = 0; j < A1 / 2; j++) q[j] = make_float4(v[2 * j].x, v[2 * j].y, v[2 * j + 1].x, v[2 * j + 1].y);
}

// The squared fields m2 become the factors of the nu step (|g_M| / |F|, MU false)
// or the mu step (|F| / |g_M|). Deep MOND is a few instructions a sample; the
// other kinds divide and take square roots in IEEE arithmetic, over a hundred
// instructions for two samples, and stay one copy in a loop that turns the
// registers round (unrolled and switched sample by sample, the passes spent
// more time on fetching instructions than on any other stall).
template <bool MU, int A1>
__device__ __forceinline__ void factors(const XArgs& a, float2* m2) {
  if (a.mu_kind == 0) {
    // from the hardware reciprocal square root (a few ulp, no IEEE divide or
    // square root): nu = sqrt(a0 / |F|) = sqrt(a0) (m2)^-1/4, mu = |g| / a0 with
    // |g| = m2 / sqrt(m2); 0 at zero field
    auto f = [&](float q) {
      const float r = q > 0.f ? rsqrtf(q) : 0.f;  // 1 / |v|
      if constexpr (MU) return q * r * a.inv_a0;
      else return a.sqrt_a0 * (r * rsqrtf(r > 0.f ? r : 1.f)) * (r > 0.f ? 1.f : 0.f);
    };
#pragma unroll
    for (int s = 0; s < A1; s++) m2[s] = make_float2(f(m2[s].x), f(m2[s].y));
    return;
  }
  auto f = [&](float q) {
    const float mag = sqrtf(q);
    return MU ? mu_factor(a.mu_kind, mag, a.a0) : nu_factor(a.mu_kind, mag, a.a0);
  };
#pragma unroll 1
  for (int s = 0; s < A1; s += 2) {
    const float2 u = make_float2(f(m2[0].x), f(m2[0].y)), w = make_float2(f(m2[1].x), f(m2[1].y));
#pragma unroll
    for (int k = 0; k < A1 - 2; k++) m2[k] = m2[k + 2];
    m2[A1 - 2] = u;
    m2[A1 - 1] = w;
  }
}

template <int N, int MODE>
__global__ void __launch_bounds__(32 * WARPS, ncomp_of(MODE) == 3 ? xctas(N) : 1) k_xreg(XArgs a) {
  using X = Geo<N>;
  constexpr int A0 = X::A0, A1 = X::A1, TL = X::TL, H = X::H, SP = X::SP, REGION = X::REGION;
  constexpr int NC = ncomp_of(MODE);
  constexpr int64_t P3 = (int64_t)N * N * N;
  extern __shared__ __align__(16) float2 xsm[];
  float2* const tw = xsm;  // N twiddles
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = lane % TL, l = lane / TL;
  // this lane's line, and its places of component 0
  const int64_t line = ((int64_t)blockIdx.x * WARPS + warp) * X::LW + l;
  float2* const sl = xsm + N + warp * NC * REGION + l * X::PITCH;
  float2* const spec = a.spec + line * SP + (NC == 1 ? blockIdx.y * a.pstride : 0);
  const int64_t rl = line * N + (NC == 1 ? (int64_t)blockIdx.y * P3 : 0);  // first real sample
  regpass::table_in(tw, a.tw, 8 * N, threadIdx.x, 32 * WARPS);
  kernel_wait();
  if constexpr (has_inv(MODE)) {
    const uint64_t pol = tma::policy_evict_first();
#pragma unroll
    for (int c = 0; c < NC; c++) {
      const float2* g = spec + c * a.pstride;
      for (int i = t; i <= H / 2; i += TL) {
        const int k = 2 * i;
        copy16_stream(sl + c * REGION + (k / A1) * X::G + k % A1, g + k, pol);
      }
    }
  }
  if (lane < 3) {
    // the real planes the pointwise stage reads, brought into L2 meanwhile (the
    // warp's lines are contiguous)
    const uint32_t rb = (uint32_t)(X::LW * N * sizeof(float));
    const int64_t o = lane * P3 + ((int64_t)blockIdx.x * WARPS + warp) * X::LW * N;
    if constexpr (MODE == X_NU || MODE == X_MU || MODE == X_NU_REAL) tma::prefetch_l2(a.gN + o, rb);
    if constexpr (MODE == X_NU_FIRST || MODE == X_NU_REAL)  // a caller's guess may lie off the prefetch's 16 bytes
      if (a.H0 && (reinterpret_cast<uintptr_t>(a.H0) & 15) == 0) tma::prefetch_l2(a.H0 + o, rb);
    if constexpr (MODE == X_NU)
      if (a.Hs_out && a.red) tma::prefetch_l2(a.Hs_out + o, rb);
  }
  tma::async_wait_all();
  __syncthreads();  // the only barrier: the twiddles
  if constexpr (has_inv(MODE)) {
#pragma unroll 1
    for (int i = t; i < NC * X::HALF; i += TL) {
      const int c = i / X::HALF, m = i - c * X::HALF;
      inv_pair<N>(sl + c * REGION, m, tw);
    }
    __syncwarp();
  }

  bool bad = false;
  float sq_dh = 0.f, sq_gn = 0.f;
#pragma unroll 1
  for (int p = t; p < A0; p += TL) {
    const int64_t rp = rl + 2 * p;  // sample pair s of this lane at rp + 2 A0 s
    float2 v[A1];
    if constexpr (MODE == X_FWD) {
#pragma unroll
      for (int s = 0; s < A1; s++) {
        v[s] = *reinterpret_cast<const float2*>(a.real_in + rp + 2 * A0 * s);
        if (a.ext_axis1 && blockIdx.y == 0) v[s] = cadd(v[s], dipole2<N>(a, line, 2 * (p + A0 * s)));
      }
      fwd_mid<N>(v, sl, p, tw);
    } else if constexpr (MODE == X_INV) {
      inv_mid<N>(v, sl, p, tw);
#pragma unroll
      for (int s = 0; s < A1; s++) {
        const int64_t ri = rp + 2 * A0 * s;
        bad |= !(isfinite(v[s].x) && isfinite(v[s].y));
        if (a.accumulate) v[s] = cadd(v[s], *reinterpret_cast<const float2*>(a.real_out + ri));
        *reinterpret_cast<float2*>(a.real_out + ri) = v[s];
        if (a.real_out2) *reinterpret_cast<float2*>(a.real_out2 + ri) = v[s];
      }
    } else {
      // F = g_N + H (nu steps) or g_M (mu step), component by component: its
      // squared length in registers, the components back to their places. The
      // real planes are requested ahead of the transform that hides them. The
      // loops over the components stay loops: unrolled, the pass is bound by
      // instruction fetch.
      float2 m2[A1], w[A1];
#pragma unroll
      for (int s = 0; s < A1; s++) m2[s] = make_float2(0.f, 0.f);
      auto request = [&](const float* f) {
#pragma unroll
        for (int s = 0; s < A1; s++) w[s] = *reinterpret_cast<const float2*>(f + 2 * A0 * s);
      };
      auto keep = [&](float* f) {
#pragma unroll
        for (int s = 0; s < A1; s++) *reinterpret_cast<float2*>(f + 2 * A0 * s) = v[s];
      };
#pragma unroll 1
      for (int c = 0; c < 3; c++) {
        float2* const sc = sl + c * REGION;
        const int64_t rc = rp + c * P3;
        if constexpr (MODE == X_NU || MODE == X_NU_REAL) {
          request(a.gN + rc);
        } else if constexpr (MODE == X_NU_FIRST) {
          if (a.H0) request(a.H0 + rc);
        }
        if constexpr (MODE != X_NU_REAL) inv_mid<N>(v, sc, p, tw);
        if constexpr (MODE == X_NU_REAL) {
#pragma unroll
          for (int s = 0; s < A1; s++) v[s] = w[s];
          if (a.H0) {
            request(a.H0 + rc);
#pragma unroll
            for (int s = 0; s < A1; s++) v[s] = cadd(v[s], w[s]);
          }
        } else if constexpr (MODE == X_NU_FIRST) {
          keep(a.gN_out + rc);  // the input is g_N
          if (a.H0) {
#pragma unroll
            for (int s = 0; s < A1; s++) v[s] = cadd(v[s], w[s]);
          }
        } else if constexpr (MODE == X_NU) {
          // the input is H after the divergence-free projection
          if (a.Hs_out) {
            if (a.red) {
#pragma unroll
              for (int s = 0; s < A1; s++) {
                const float2 d = csub(v[s], *reinterpret_cast<const float2*>(a.Hs_out + rc + 2 * A0 * s));
                sq_dh += d.x * d.x + d.y * d.y;
                sq_gn += w[s].x * w[s].x + w[s].y * w[s].y;
              }
            }
            keep(a.Hs_out + rc);
          }
#pragma unroll
          for (int s = 0; s < A1; s++) v[s] = cadd(v[s], w[s]);
        } else {
          if (a.gM_out) keep(a.gM_out + rc);
        }
        float4* const q = reinterpret_cast<float4*>(sc + p * X::G);
#pragma unroll
        for (int j = 0; j < A1 / 2; j++) q[j] = make_float4(v[2 * j].x, v[2 * j].y, v[2 * j + 1].x, v[2 * j + 1].y);
#pragma unroll
        for (int s = 0; s < A1; s++) {
          m2[s].x = fmaf(v[s].x, v[s].x, m2[s].x);
          m2[s].y = fmaf(v[s].y, v[s].y, m2[s].y);
        }
      }
#pragma unroll
      for (int s = 0; s < A1; s++) bad |= !(isfinite(m2[s].x) && isfinite(m2[s].y));
      factors<MODE == X_MU, A1>(a, m2);
#pragma unroll 1
      for (int c = 0; c < 3; c++) {
        float2* const sc = sl + c * REGION;
        if constexpr (MODE == X_MU) request(a.gN + rp + c * P3);
        const float4* const q = reinterpret_cast<const float4*>(sc + p * X::G);
#pragma unroll
        for (int j = 0; j < A1 / 2; j++) {
          const float4 f = q[j];
          v[2 * j] = make_float2(f.x * m2[2 * j].x, f.y * m2[2 * j].y);
          v[2 * j + 1] = make_float2(f.z * m2[2 * j + 1].x, f.w * m2[2 * j + 1].y);
        }
        if constexpr (MODE == X_MU) {
#pragma unroll
          for (int s = 0; s < A1; s++) v[s] = csub(v[s], w[s]);  // H = F - g_N
        }
        fwd_mid<N>(v, sc, p, tw);
      }
    }
  }
  if (bad) set_status(a.status, ST_NAN);
  if (MODE == X_NU && a.red && a.Hs_out) {
    for (int o = 16; o > 0; o >>= 1) {
      sq_dh += __shfl_xor_sync(0xffffffffu, sq_dh, o);
      sq_gn += __shfl_xor_sync(0xffffffffu, sq_gn, o);
    }
    if (lane == 0) {
      atomicAdd(a.red, (double)sq_dh);
      atomicAdd(a.red + 1, (double)sq_gn);
    }
  }
  if constexpr (has_fwd(MODE)) {
    __syncwarp();
#pragma unroll 1
    for (int i = t; i < NC * X::HALF; i += TL) {
      const int c = i / X::HALF, m = i - c * X::HALF;
      fwd_pair<N>(sl + c * REGION, m, tw, spec + c * a.pstride);
    }
  }
}

}  // namespace xreg
