// fno_dft.cuh -- the truncated transforms of the surrogate's spectral layers:
// only M modes per axis are kept (x: real -> kx < M; y and z: frequencies
// -M .. M-1, stored as f and 2M - f), so each axis is a small contraction.
//
// Positions x and n - x share their cosines and their sines up to a sign, and
// so do the frequencies f and -f: with the sum a and the difference b of such
// a pair, sum_x v e^{-i t f x} = A - iB and, for -f, A + iB, where A = sum a
// cos and B = sum b sin over half the positions. Every contraction here runs
// over the folded half and yields a pair of outputs, which leaves a quarter
// of the multiplications along a complex axis and half of them along the real
// one, done two at a time (fma.rn.f32x2). n <= 64 is a multiple of 4, 2M <= n.
//
// Kernels take bounds n <= NX and M <= MX; FULL: they are n and M themselves
// (the sides in common use), so that no inner step is conditional.
#pragma once

namespace dft {

constexpr int TH = 256;

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long&>(r))
      : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)),
        "l"(reinterpret_cast<unsigned long long&>(c)));
  return r;
}
__device__ __forceinline__ float2 lo(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi(const float4& v) { return make_float2(v.z, v.w); }

// (cos, sin)(2 pi m/n), m < n, into shared memory; the caller synchronises.
__device__ __forceinline__ void circle(float2* cs, int n) {
  if ((int)threadIdx.x < n) {
    float s, c;
    sincospif(2.0f * (float)threadIdx.x / (float)n, &s, &c);
    cs[threadIdx.x] = make_float2(c, s);
  }
}
// T[y][f] = (c, c, s, s)(2 pi f y/n), y < rows, f <= M (doubled for the packed products).
__device__ __forceinline__ void pair_table(float4* T, const float2* cs, int rows, int n, int M) {
  for (int e = threadIdx.x; e < rows * (M + 1); e += TH) {
    const float2 w = cs[(e / (M + 1)) * (e % (M + 1)) % n];
    T[e] = make_float4(w.x, w.x, w.y, w.y);
  }
}

// Forward along x and y of one plane at a time, v [n][n] real -> out [2M][M].
// The plane's rows are folded on their way into shared memory (the next
// plane's loads are in flight meanwhile); x: a lane owns one kx with its table
// column in registers and takes the rows y and n - y together, so the result
// is folded along y too; y: a thread owns one kx and FB frequency pairs.
// Bound by shared memory (broadcast reads, 86% of its pipe). 32 channels: 64^3,
// M = 16: 56 us with the unfolded sums, 32 us folded, 24 us with the bounds
// fixed; 32^3: 16.6 -> 7.3 us.
__host__ __device__ inline size_t smem_xy_fwd(int n, int M) {
  return sizeof(float2) * 64 + sizeof(float) * n * (n + 4) + sizeof(float4) * ((size_t)n / 2 * M + n / 2 * (M + 1));
}
template <int NX, int MX, bool FULL>
__global__ void __launch_bounds__(TH, 2) k_xy_fwd(const float* __restrict__ v, float2* __restrict__ out, int n_, int M_,
                                                  int nplanes) {
  constexpr int HX = NX / 2, FIT = NX * HX / TH ? NX * HX / TH : 1, RP = 32 / MX, FB = 2;
  extern __shared__ __align__(16) float4 sm4[];
  const int n = FULL ? NX : n_, M = FULL ? MX : M_;
  const int H = n / 2, PF = n + 4, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float4* sX = sm4;                                      // [H][M] (sum, difference) of the rows y and n - y
  float4* sT = sX + H * M;                               // [H][M + 1]
  float* sF = reinterpret_cast<float*>(sT + H * (M + 1));  // [n][PF]: H pairs (sum, difference) of x and n - x
  float2* cs = reinterpret_cast<float2*>(sF + n * PF);
  circle(cs, n);
  __syncthreads();
  pair_table(sT, cs, H, n, M);
  const int kx = lane % MX;
  float2 tx[HX];
#pragma unroll
  for (int x = 1; x < HX; x++) {
    const float2 w = (x < H && kx < M) ? cs[kx * x % n] : make_float2(0.f, 0.f);
    tx[x] = make_float2(w.x, -w.y);
  }
  const int fx = tid % HX, fx2 = fx ? n - fx : H, fy = tid / HX;  // this thread's elements of the fold
  float pre[FIT][2];
  auto fetch = [&](int plane) {
    const float* src = v + (int64_t)plane * n * n;
#pragma unroll
    for (int k = 0; k < FIT; k++) {
      const int y = fy + k * (TH / HX);
      if (fx < H && y < n) {
        pre[k][0] = src[y * n + fx];
        pre[k][1] = src[y * n + fx2];
      }
    }
  };
  kernel_wait();
  v = after_wait(v);
  if ((int)blockIdx.x < nplanes) fetch(blockIdx.x);
  for (int plane = blockIdx.x; plane < nplanes; plane += gridDim.x) {
#pragma unroll
    for (int k = 0; k < FIT; k++) {
      const int y = fy + k * (TH / HX);
      if (fx < H && y < n)
        *reinterpret_cast<float2*>(sF + y * PF + 2 * fx) =
            make_float2(pre[k][0] + pre[k][1], pre[k][0] - pre[k][1]);
    }
    if (plane + (int)gridDim.x < nplanes) fetch(plane + gridDim.x);
    __syncthreads();
    for (int r = warp * RP + lane / MX; r < H; r += 8 * RP) {
      const float4* a = reinterpret_cast<const float4*>(sF + r * PF);
      const float4* b = reinterpret_cast<const float4*>(sF + (r ? n - r : H) * PF);
      float2 p[2], q[2];
      {  // the pair x = 0, n/2 holds (v0 + vH, v0 - vH): the sums of the even and of the odd kx
        const float4 u = a[0], w = b[0];
        p[0] = make_float2((kx & 1) ? u.y : u.x, 0.f);
        q[0] = make_float2((kx & 1) ? w.y : w.x, 0.f);
        p[1] = fma2(hi(u), tx[1], make_float2(0.f, 0.f));
        q[1] = fma2(hi(w), tx[1], make_float2(0.f, 0.f));
      }
#pragma unroll
      for (int x = 2; x < HX; x += 2)
        if (x < H) {
          const float4 u = a[x / 2], w = b[x / 2];
          p[0] = fma2(lo(u), tx[x], p[0]);
          q[0] = fma2(lo(w), tx[x], q[0]);
          p[1] = fma2(hi(u), tx[x + 1], p[1]);
          q[1] = fma2(hi(w), tx[x + 1], q[1]);
        }
      p[0].x += p[1].x;
      p[0].y += p[1].y;
      q[0].x += q[1].x;
      q[0].y += q[1].y;
      if (kx < M) sX[r * M + kx] = make_float4(p[0].x + q[0].x, p[0].y + q[0].y, p[0].x - q[0].x, p[0].y - q[0].y);
    }
    __syncthreads();
    float2* o = out + (int64_t)plane * 2 * M * M;
    for (int t = tid; t < ((M + FB) / FB) * M; t += TH) {
      const int k = t % M, f0 = (t / M) * FB;
      float2 A[FB], B[FB];
      const float4 ab0 = sX[k];
      int fo[FB];
#pragma unroll
      for (int j = 0; j < FB; j++) {
        fo[j] = min(f0 + j, M);
        A[j] = (fo[j] & 1) ? hi(ab0) : lo(ab0);
        B[j] = make_float2(0.f, 0.f);
      }
#pragma unroll 4
      for (int y = 1; y < H; y++) {
        const float4 ab = sX[y * M + k];
#pragma unroll
        for (int j = 0; j < FB; j++) {
          const float4 w = sT[y * (M + 1) + fo[j]];
          A[j] = fma2(lo(ab), lo(w), A[j]);
          B[j] = fma2(hi(ab), hi(w), B[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < FB; j++) {
        const int f = f0 + j;
        if (f < M) o[f * M + k] = make_float2(A[j].x + B[j].y, A[j].y - B[j].x);
        if (f > 0 && f <= M) o[(2 * M - f) * M + k] = make_float2(A[j].x - B[j].y, A[j].y + B[j].x);
      }
    }
  }
}

// Folded half of 2M frequencies: slot f holds (in[f] + in[-f], in[f] - in[-f])
// for 0 < f < M; slot 0 has in[0] alone and slot M has in[-M] alone. The
// thread that has (f, -f), or (0, -M) as p and q, writes its slots.
__device__ __forceinline__ void fold_freq(float4* s, int pitch, int f, int M, float2 p, float2 q) {
  if (f) {
    s[f * pitch] = make_float4(p.x + q.x, p.y + q.y, p.x - q.x, p.y - q.y);
  } else {
    s[0] = make_float4(p.x, p.y, 0.f, 0.f);
    s[M * pitch] = make_float4(q.x, q.y, -q.x, -q.y);
  }
}

// Inverse along y and x of one plane at a time, in [2M][M] -> real [n][n],
// added into z; then v = gelu(z) (act 1), v = z (act 2) or nothing. The x sum
// takes the weight w0 at kx = 0 and w1 elsewhere. y: a thread owns one kx and
// YB position pairs; x: a lane owns the positions x and n - x with its table
// column in registers (lane 0: the positions 0 and n/2). Bound by latency and
// by shared memory (73% of its pipe) with two CTAs per SM. 32 channels: 64^3,
// M = 16: 112 us unfolded, 48 us folded, 36 us with the bounds fixed; 32^3:
// 25 -> 9.0 us.
__host__ __device__ inline size_t smem_xy_inv(int n, int M) {
  return sizeof(float2) * 64 + sizeof(float) * n * (2 * ((M + 1) & ~1) + 4) +
         sizeof(float4) * ((size_t)(M + 1) * M + (n / 2 + 1) * (M + 1));
}
template <int NX, int MX, bool FULL>
__global__ void __launch_bounds__(TH, 2) k_xy_inv(const float2* __restrict__ in, float* __restrict__ z,
                                                  float* __restrict__ v, int n_, int M_, float w0, float w1, int act,
                                                  int nplanes) {
  constexpr int LX = NX / 2, RW = 32 / LX, NK = NX / (8 * RW) ? NX / (8 * RW) : 1;
  constexpr int FIT = MX * MX / TH ? MX * MX / TH : 1, YB = NX > 32 ? 3 : 2;
  extern __shared__ __align__(16) float4 sm4[];
  const int n = FULL ? NX : n_, M = FULL ? MX : M_;
  const int H = n / 2, Me = (M + 1) & ~1, XS = 2 * Me + 4, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float4* sI = sm4;                                              // [M + 1][M], folded
  float4* sT = sI + (M + 1) * M;                                 // [H + 1][M + 1]
  float* sX = reinterpret_cast<float*>(sT + (H + 1) * (M + 1));  // [n][XS]
  float2* cs = reinterpret_cast<float2*>(sX + n * XS);
  circle(cs, n);
  for (int e = tid; e < n * XS; e += TH) sX[e] = 0.f;  // the column past an odd M is read, times 0
  __syncthreads();
  pair_table(sT, cs, H + 1, n, M);
  const int x = lane % LX, x2 = x ? n - x : H, sub = lane / LX;
  float2 tt[MX];
#pragma unroll
  for (int k = 0; k < MX; k++) {
    const float2 w = (k < M && x < H) ? cs[k * x % n] : make_float2(0.f, 0.f);
    tt[k] = make_float2(w.x * (k ? w1 : w0), -w.y * (k ? w1 : w0));
  }
  const int fk = tid % MX, ff = tid / MX;  // this thread's elements of the fold
  float2 pre[FIT][2];
  auto fetch = [&](int plane) {
    const float2* src = in + (int64_t)plane * 2 * M * M;
#pragma unroll
    for (int k = 0; k < FIT; k++) {
      const int f = ff + k * (TH / MX);
      if (fk < M && f < M) {
        pre[k][0] = src[f * M + fk];
        pre[k][1] = src[(f ? 2 * M - f : M) * M + fk];
      }
    }
  };
  kernel_wait();
  in = after_wait(in);
  z = after_wait(z);
  if ((int)blockIdx.x < nplanes) fetch(blockIdx.x);
  for (int plane = blockIdx.x; plane < nplanes; plane += gridDim.x) {
#pragma unroll
    for (int k = 0; k < FIT; k++) {
      const int f = ff + k * (TH / MX);
      if (fk < M && f < M) fold_freq(sI + fk, M, f, M, pre[k][0], pre[k][1]);
    }
    if (plane + (int)gridDim.x < nplanes) fetch(plane + gridDim.x);
    // this thread's values of z, in flight during the y sum
    float* zp = z + (int64_t)plane * n * n;
    float* vp = v ? v + (int64_t)plane * n * n : nullptr;
    float zr[NK][2];
#pragma unroll
    for (int k = 0; k < NK; k++) {
      const int y = (warp + 8 * k) * RW + sub;
      if (y < n && x < H) {
        zr[k][0] = zp[y * n + x];
        zr[k][1] = zp[y * n + x2];
      }
    }
    __syncthreads();
    for (int t = tid; t < ((H + YB) / YB) * M; t += TH) {
      const int k = t % M, y0 = (t / M) * YB;
      float2 A[YB], B[YB];
      int yo[YB];
#pragma unroll
      for (int j = 0; j < YB; j++) {
        yo[j] = min(y0 + j, H) * (M + 1);
        A[j] = B[j] = make_float2(0.f, 0.f);
      }
#pragma unroll 4
      for (int f = 0; f <= M; f++) {
        const float4 ab = sI[f * M + k];
#pragma unroll
        for (int j = 0; j < YB; j++) {
          const float4 w = sT[yo[j] + f];
          A[j] = fma2(lo(ab), lo(w), A[j]);
          B[j] = fma2(hi(ab), hi(w), B[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < YB; j++) {
        const int y = y0 + j;
        if (y <= H) *reinterpret_cast<float2*>(sX + y * XS + 2 * k) = make_float2(A[j].x - B[j].y, A[j].y + B[j].x);
        if (y > 0 && y < H)
          *reinterpret_cast<float2*>(sX + (n - y) * XS + 2 * k) = make_float2(A[j].x + B[j].y, A[j].y - B[j].x);
      }
    }
    __syncthreads();
    // x = n/2 of this warp's rows, a row per lane: the cosines are +-1
    float xh = 0.f;
    {
      const int y = (warp + 8 * (lane / RW)) * RW + lane % RW;
      if (lane < NK * RW && y < n) {
        const float4* xr = reinterpret_cast<const float4*>(sX + y * XS);
        float e = 0.f;
#pragma unroll
        for (int q = 0; q < MX / 2; q++)
          if (2 * q < M) {
            const float4 u = xr[q];
            if (q == 0) xh = w0 * u.x;
            else e += u.x;
            e -= u.z;
          }
        xh = fmaf(w1, e, xh);
      }
    }
#pragma unroll
    for (int k = 0; k < NK; k++) {
      const int y = (warp + 8 * k) * RW + sub;
      const float h = __shfl_sync(0xffffffffu, xh, k * RW + sub);
      if (y < n && x < H) {
        const float4* xr = reinterpret_cast<const float4*>(sX + y * XS);
        float2 e0 = make_float2(0.f, 0.f), e1 = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < MX / 2; q++)
          if (2 * q < M) {
            const float4 u = xr[q];
            e0 = fma2(lo(u), tt[2 * q], e0);
            e1 = fma2(hi(u), tt[2 * q + 1], e1);
          }
        const float E = e0.x + e1.x, O = e0.y + e1.y;
        const float za = zr[k][0] + (E + O), zb = zr[k][1] + (x ? E - O : h);
        zp[y * n + x] = za;
        zp[y * n + x2] = zb;
        if (act == 1) {
          vp[y * n + x] = gelu_t(za, nullptr);
          vp[y * n + x2] = gelu_t(zb, nullptr);
        } else if (act == 2) {
          vp[y * n + x] = za;
          vp[y * n + x2] = zb;
        }
      }
    }
  }
}

// Along z, 32 columns of one channel per CTA: a warp owns FB (YB) folded
// outputs of all 32 columns, a lane a column. Few enough CTAs that all are
// resident at once. 64^3, M = 16, 32 channels: 22.8 (forward) and 17.0 us
// (inverse) unfolded -> 8.1 and 7.7 us; 32^3: 12.3 -> 5.7 us.
constexpr int ZC = 32;
__host__ __device__ inline size_t smem_z(int n, int M, int slots, int rows) {
  return sizeof(float2) * 64 + sizeof(float4) * ((size_t)slots * ZC + rows * (M + 1));
}
// in [c][n][I] -> out [c][2M][I]
template <int NX, int MX, bool FULL>
__global__ void __launch_bounds__(TH) k_z_fwd(const float2* __restrict__ in, float2* __restrict__ out, int n_, int M_,
                                              int I) {
  constexpr int FB = MX / 8 + 1;
  extern __shared__ __align__(16) float4 sm4[];
  const int n = FULL ? NX : n_, M = FULL ? MX : M_;
  const int H = n / 2, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * ZC + lane;
  float4* sA = sm4;         // [H][ZC]
  float4* sT = sA + H * ZC;  // [H][M + 1]
  float2* cs = reinterpret_cast<float2*>(sT + H * (M + 1));
  in += (int64_t)blockIdx.y * n * I;
  out += (int64_t)blockIdx.y * 2 * M * I;
  circle(cs, n);
  kernel_wait();
  in = after_wait(in);
  float2 p[4], q[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int z = warp + 8 * k;
    p[k] = q[k] = make_float2(0.f, 0.f);
    if (z < H && i < I) {
      p[k] = in[(int64_t)z * I + i];
      q[k] = in[(int64_t)(z ? n - z : H) * I + i];
    }
  }
  __syncthreads();
  pair_table(sT, cs, H, n, M);
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int z = warp + 8 * k;
    if (z < H) sA[z * ZC + lane] = make_float4(p[k].x + q[k].x, p[k].y + q[k].y, p[k].x - q[k].x, p[k].y - q[k].y);
  }
  __syncthreads();
  const int f0 = warp * FB;
  if (f0 > M || i >= I) return;
  float2 A[FB], B[FB];
  int fo[FB];
  const float4 ab0 = sA[lane];
#pragma unroll
  for (int j = 0; j < FB; j++) {
    fo[j] = min(f0 + j, M);
    A[j] = (fo[j] & 1) ? hi(ab0) : lo(ab0);
    B[j] = make_float2(0.f, 0.f);
  }
#pragma unroll 4
  for (int z = 1; z < H; z++) {
    const float4 ab = sA[z * ZC + lane];
#pragma unroll
    for (int j = 0; j < FB; j++) {
      const float4 w = sT[z * (M + 1) + fo[j]];
      A[j] = fma2(lo(ab), lo(w), A[j]);
      B[j] = fma2(hi(ab), hi(w), B[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < FB; j++) {
    const int f = f0 + j;
    if (f < M) out[(int64_t)f * I + i] = make_float2(A[j].x + B[j].y, A[j].y - B[j].x);
    if (f > 0 && f <= M) out[(int64_t)(2 * M - f) * I + i] = make_float2(A[j].x - B[j].y, A[j].y + B[j].x);
  }
}
// in [c][2M][I] -> out [c][n][I]
template <int NX, int MX, bool FULL>
__global__ void __launch_bounds__(TH) k_z_inv(const float2* __restrict__ in, float2* __restrict__ out, int n_, int M_,
                                              int I) {
  constexpr int YB = NX / 16 + 1;
  extern __shared__ __align__(16) float4 sm4[];
  const int n = FULL ? NX : n_, M = FULL ? MX : M_;
  const int H = n / 2, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * ZC + lane;
  float4* sA = sm4;               // [M + 1][ZC]
  float4* sT = sA + (M + 1) * ZC;  // [H + 1][M + 1]
  float2* cs = reinterpret_cast<float2*>(sT + (H + 1) * (M + 1));
  in += (int64_t)blockIdx.y * 2 * M * I;
  out += (int64_t)blockIdx.y * n * I;
  circle(cs, n);
  kernel_wait();
  in = after_wait(in);
  float2 p[4], q[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int f = warp + 8 * k;
    p[k] = q[k] = make_float2(0.f, 0.f);
    if (f < M && i < I) {
      p[k] = in[(int64_t)f * I + i];
      q[k] = in[(int64_t)(f ? 2 * M - f : M) * I + i];
    }
  }
  __syncthreads();
  pair_table(sT, cs, H + 1, n, M);
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int f = warp + 8 * k;
    if (f < M) fold_freq(sA + lane, ZC, f, M, p[k], q[k]);
  }
  __syncthreads();
  const int y0 = warp * YB;
  if (y0 > H || i >= I) return;
  float2 A[YB], B[YB];
  int yo[YB];
#pragma unroll
  for (int j = 0; j < YB; j++) {
    yo[j] = min(y0 + j, H) * (M + 1);
    A[j] = B[j] = make_float2(0.f, 0.f);
  }
#pragma unroll 4
  for (int f = 0; f <= M; f++) {
    const float4 ab = sA[f * ZC + lane];
#pragma unroll
    for (int j = 0; j < YB; j++) {
      const float4 w = sT[yo[j] + f];
      A[j] = fma2(lo(ab), lo(w), A[j]);
      B[j] = fma2(hi(ab), hi(w), B[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < YB; j++) {
    const int y = y0 + j;
    if (y <= H) out[(int64_t)y * I + i] = make_float2(A[j].x - B[j].y, A[j].y + B[j].x);
    if (y > 0 && y < H) out[(int64_t)(n - y) * I + i] = make_float2(A[j].x + B[j].y, A[j].y - B[j].x);
  }
}

}  // namespace dft
