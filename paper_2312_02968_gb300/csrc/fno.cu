// fno.cu -- the learned warm start (include/mond_fno.h): a Fourier neural
// operator on a coarse grid, forward and backward, BF16 weights with FP32
// accumulation, plus the kernels that move fields between the solver mesh and
// the network grid and the sphere-mixture density used to make training pairs.
//
// The spectral convolution keeps only M modes per axis, so its forward and
// inverse transforms are truncated DFTs, evaluated as one small contraction
// per axis (x: real -> M complex; y, z: n -> 2M). The inverse with weight 1
// and no 1/n^3 is the adjoint of the forward, which the backward pass uses.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "../../include/mond_fno.h"
#include "common.cuh"
#include "internal.h"

namespace {

constexpr int TB = 256;

struct Shape {
  int n, C, M, L;
  int64_t V;  // n^3
  int K;      // M (2M)(2M)
  __host__ __device__ int64_t layer_size() const { return (int64_t)C * C + C + 2LL * K * C * C; }
  __host__ __device__ int64_t off_P() const { return 0; }
  __host__ __device__ int64_t off_p() const { return 4LL * C; }
  __host__ __device__ int64_t off_layer(int l) const { return 5LL * C + l * layer_size(); }
  __host__ __device__ int64_t off_W(int l) const { return off_layer(l); }
  __host__ __device__ int64_t off_b(int l) const { return off_layer(l) + (int64_t)C * C; }
  __host__ __device__ int64_t off_R(int l) const { return off_layer(l) + (int64_t)C * C + C; }
  __host__ __device__ int64_t off_Q() const { return off_layer(L); }
  __host__ __device__ int64_t off_q() const { return off_Q() + 3LL * C; }
  __host__ __device__ int64_t count() const { return off_q() + 3; }
};

bool make_shape(const mond_fno_shape& s, Shape* o) {
  if (s.n < 8 || s.n > 64 || s.n % 4 || s.width < 2 || s.width > 32 || s.width % 2 || s.modes < 1 ||
      2 * s.modes > s.n ||
      s.layers < 1 || s.layers > 8)
    return false;
  o->n = s.n;
  o->C = s.width;
  o->M = s.modes;
  o->L = s.layers;
  o->V = (int64_t)s.n * s.n * s.n;
  o->K = s.modes * 4 * s.modes * s.modes;
  return true;
}

// Workspace layout for one sample.
struct Work {
  float* v;      // (L+1) x C x V activations (v_0 .. v_L)
  float* z;      // L x C x V pre-activations
  float2* shat;  // L x C x K truncated spectra of v_l
  float2* b;     // C x n x 2M x M (x- and y-transformed planes)
  float2* c;     // C x K          (z-transformed / mixed)
  float2* d;     // C x K
  float* dv;     // C x V
  float* dv2;    // C x V
  float* dz;     // C x V
};

size_t carve(const Shape& s, char* base, Work* w) {
  size_t off = 0;
  auto take = [&](size_t bytes) -> char* {
    char* p = base ? base + off : nullptr;
    off += (bytes + 255) & ~(size_t)255;
    return p;
  };
  const size_t CV = (size_t)s.C * s.V;
  Work t{};
  t.v = (float*)take(sizeof(float) * CV * (s.L + 1));
  t.z = (float*)take(sizeof(float) * CV * s.L);
  t.shat = (float2*)take(sizeof(float2) * (size_t)s.C * s.K * s.L);
  t.b = (float2*)take(sizeof(float2) * (size_t)s.C * s.n * 2 * s.M * s.M);
  t.c = (float2*)take(sizeof(float2) * (size_t)s.C * s.K);
  t.d = (float2*)take(sizeof(float2) * (size_t)s.C * s.K);
  t.dv = (float*)take(sizeof(float) * CV);
  t.dv2 = (float*)take(sizeof(float) * CV);
  t.dz = (float*)take(sizeof(float) * CV);
  if (w) *w = t;
  return off;
}

__device__ __forceinline__ float bf(const uint16_t* p, int64_t i) {
  return __bfloat162float(__ushort_as_bfloat16(p[i]));
}

// out[o][v] = sum_i W[o][i] in[i][v] (+ b[o]); transpose uses W[i][o].
// CMAX >= Cin: the input channels sit in registers, the weights in shared
// memory zero-padded to CMAX columns.
template <int CMAX>
__global__ void __launch_bounds__(256) k_pw(const float* __restrict__ in, int Cin, const uint16_t* __restrict__ W,
                                            const uint16_t* __restrict__ b, int Cout, float* __restrict__ out,
                                            int64_t V, int transpose) {
  kernel_wait();
  in = after_wait(in);
  W = after_wait(W);
  b = after_wait(b);
  __shared__ __align__(16) float sW[32 * CMAX];
  __shared__ float sb[32];
  for (int e = threadIdx.x; e < Cout * CMAX; e += blockDim.x) {
    const int o = e / CMAX, i = e % CMAX;
    sW[e] = i < Cin ? (transpose ? bf(W, (int64_t)i * Cout + o) : bf(W, (int64_t)o * Cin + i)) : 0.f;
  }
  for (int o = threadIdx.x; o < Cout; o += blockDim.x) sb[o] = b ? bf(b, o) : 0.f;
  __syncthreads();
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
    float x[CMAX];
#pragma unroll
    for (int i = 0; i < CMAX; i++) x[i] = i < Cin ? in[i * V + v] : 0.f;
    for (int o = 0; o < Cout; o++) {
      float acc = sb[o];
      const float4* w4 = reinterpret_cast<const float4*>(sW + o * CMAX);
#pragma unroll
      for (int i = 0; i < CMAX / 4; i++) {
        const float4 w = w4[i];
        acc = fmaf(w.x, x[4 * i], acc);
        acc = fmaf(w.y, x[4 * i + 1], acc);
        acc = fmaf(w.z, x[4 * i + 2], acc);
        acc = fmaf(w.w, x[4 * i + 3], acc);
      }
      out[o * V + v] = acc;
    }
  }
}

// The same channel mixing on the tensor cores (mma.sync m16n8k16, bfloat16
// operands, FP32 accumulation), for Cin, Cout <= 32: out[o][v] = sum_i W[o][i]
// in[i][v] (+ b[o]); transpose uses W[i][o]. The weights are bfloat16 already;
// each FP32 input is split into three bfloat16 parts x = h + m + l (the top,
// middle and low eight bits of its significand), so the three products per
// weight are exact and only the FP32 accumulation rounds, as in the FMA chain
// of k_pw.
// Bound by memory: a warp takes 32 voxels a step, as four 8-column tiles whose
// columns are interleaved (column g of tile t is voxel 4g + t), so that a lane
// loads four neighbouring voxels of a channel at once, all eight of its
// channels before any is used, and stores four. One warp of 8 voxels with
// 4-byte accesses: 37 us for 64^3, 32 -> 32 channels (67 MB); now 16.4 us.
__device__ __forceinline__ uint32_t pack_bf16(float lo_half, float hi_half) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(lo_half, hi_half);
  return *reinterpret_cast<const uint32_t*>(&p);
}
__device__ __forceinline__ float lo_bf16(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float hi_bf16(uint32_t p) { return __uint_as_float(p & 0xffff0000u); }
__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int MT>  // Cout <= 16 MT
__global__ void __launch_bounds__(256, 2) k_pw_mma(const float* __restrict__ in, int Cin,
                                                   const uint16_t* __restrict__ W, const uint16_t* __restrict__ b,
                                                   int Cout, float* __restrict__ out, int64_t V, int transpose,
                                                   int vec_out) {
  kernel_wait();
  in = after_wait(in);
  W = after_wait(W);
  b = after_wait(b);
  __shared__ uint16_t sW[32][32 + 8];  // [o][i], zero-padded; row pitch 80 bytes (conflict-free fragments)
  __shared__ float sb[32];
  for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x) {
    const int o = e / 32, i = e % 32;
    uint16_t w = 0;
    if (o < Cout && i < Cin) w = transpose ? W[(int64_t)i * Cout + o] : W[(int64_t)o * Cin + i];
    sW[o][i] = w;
  }
  for (int o = threadIdx.x; o < 32; o += blockDim.x) sb[o] = (b && o < Cout) ? bf(b, o) : 0.f;
  __syncthreads();
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  // A fragments: [M tile][K step][4 registers], row-major 16x16 tiles of sW
  uint32_t A[MT][2][4];
#pragma unroll
  for (int mt = 0; mt < MT; mt++)
#pragma unroll
    for (int ks = 0; ks < 2; ks++) {
      const int r0 = 16 * mt + g, c0 = 16 * ks + 2 * q;
      A[mt][ks][0] = *reinterpret_cast<const uint32_t*>(&sW[r0][c0]);
      A[mt][ks][1] = *reinterpret_cast<const uint32_t*>(&sW[r0 + 8][c0]);
      A[mt][ks][2] = *reinterpret_cast<const uint32_t*>(&sW[r0][c0 + 8]);
      A[mt][ks][3] = *reinterpret_cast<const uint32_t*>(&sW[r0 + 8][c0 + 8]);
    }
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; v0 < V; v0 += warps * 32) {
    // rows k = 16 ks + 8 rr + 2 q + j of the B fragments, four voxels of each
    float4 x[2][2][2];
#pragma unroll
    for (int ks = 0; ks < 2; ks++)
#pragma unroll
      for (int rr = 0; rr < 2; rr++)
#pragma unroll
        for (int j = 0; j < 2; j++) {
          const int k = 16 * ks + 8 * rr + 2 * q + j;
          x[ks][rr][j] = k < Cin ? *(reinterpret_cast<const float4*>(in + (int64_t)k * V + v0) + g)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    float d[MT][4][4];  // [M tile][voxel tile][C fragment: rows g, g + 8, columns 2q, 2q + 1]
#pragma unroll
    for (int t = 0; t < 4; t++) {
      uint32_t Bh[2][2], Bm[2][2], Bl[2][2];
#pragma unroll
      for (int ks = 0; ks < 2; ks++)
#pragma unroll
        for (int rr = 0; rr < 2; rr++) {
          const float* f0 = &x[ks][rr][0].x;
          const float* f1 = &x[ks][rr][1].x;
          Bh[ks][rr] = pack_bf16(f0[t], f1[t]);
          const float r0 = f0[t] - lo_bf16(Bh[ks][rr]), r1 = f1[t] - hi_bf16(Bh[ks][rr]);  // exact
          Bm[ks][rr] = pack_bf16(r0, r1);
          Bl[ks][rr] = pack_bf16(r0 - lo_bf16(Bm[ks][rr]), r1 - hi_bf16(Bm[ks][rr]));  // exact, a bfloat16
        }
#pragma unroll
      for (int mt = 0; mt < MT; mt++) {
        d[mt][t][0] = d[mt][t][1] = sb[16 * mt + g];
        d[mt][t][2] = d[mt][t][3] = sb[16 * mt + g + 8];
#pragma unroll
        for (int ks = 0; ks < 2; ks++) {
          mma_bf16(d[mt][t], A[mt][ks], Bl[ks][0], Bl[ks][1]);  // smallest parts first
          mma_bf16(d[mt][t], A[mt][ks], Bm[ks][0], Bm[ks][1]);
          mma_bf16(d[mt][t], A[mt][ks], Bh[ks][0], Bh[ks][1]);
        }
      }
    }
#pragma unroll
    for (int mt = 0; mt < MT; mt++)
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const int o = 16 * mt + g + 8 * (e >> 1);
        if (o >= Cout) continue;
        float* p = out + (int64_t)o * V + v0 + 8 * q + 4 * (e & 1);
        if (vec_out) {
          *reinterpret_cast<float4*>(p) = make_float4(d[mt][0][e], d[mt][1][e], d[mt][2][e], d[mt][3][e]);
        } else {
#pragma unroll
          for (int t = 0; t < 4; t++) p[t] = d[mt][t][e];
        }
      }
  }
}

// dW[o][i] += sum_v dout[o][v] in[i][v]; db[o] += sum_v dout[o][v].
// Tiles of 64 voxels in shared memory, the next one's loads in flight; a
// thread owns the rows ob, ob + 16 and the columns ib, ib + 16 of dW, four
// voxels a read. A tile is summed by itself and then added to the running sums,
// so that a chain of additions is 64 long and not 64 times the CTA's tiles. A
// CTA per SM: each adds its 1056 sums to the same words, and with four CTAs per
// SM those atomics and one product per two reads took 16.5 us at 32^3 (32 x 32
// channels); now 9.0 us.
__global__ void __launch_bounds__(256) k_wgrad(const float* __restrict__ dout, int Cout, const float* __restrict__ in,
                                               int Cin, int64_t V, float* dW, float* db, int vec) {
  kernel_wait();
  dout = after_wait(dout);
  in = after_wait(in);
  constexpr int CH = 64, P = CH + 4;
  __shared__ __align__(16) float so[32 * P], si[32 * P];
  const int tid = threadIdx.x, ob = tid >> 4, ib = tid & 15, ntiles = (int)(V / CH);
  float4 pre[4];
  auto fetch = [&](int tile) {
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const int row = (tid >> 4) + 16 * (k & 1);
      const float* src = k < 2 ? dout : in;
      const bool live = row < (k < 2 ? Cout : Cin);
      const float* p = src + (int64_t)row * V + (int64_t)tile * CH + 4 * (tid & 15);
      if (!live) pre[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      else if (vec) pre[k] = *(reinterpret_cast<const float4*>(p));
      else pre[k] = make_float4(*(p), *(p + 1), *(p + 2), *(p + 3));
    }
  };
  float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, bias[2] = {0.f, 0.f};
  if ((int)blockIdx.x < ntiles) fetch(blockIdx.x);
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; k++)
      *reinterpret_cast<float4*>((k < 2 ? so : si) + ((tid >> 4) + 16 * (k & 1)) * P + 4 * (tid & 15)) = pre[k];
    __syncthreads();
    if (tile + (int)gridDim.x < ntiles) fetch(tile + gridDim.x);
    float s[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, sb[2] = {0.f, 0.f};
#pragma unroll 4
    for (int c = 0; c < CH; c += 4) {
      float4 a[2], x[2];
#pragma unroll
      for (int r = 0; r < 2; r++) {
        a[r] = *reinterpret_cast<const float4*>(so + (ob + 16 * r) * P + c);
        x[r] = *reinterpret_cast<const float4*>(si + (ib + 16 * r) * P + c);
        sb[r] += (a[r].x + a[r].y) + (a[r].z + a[r].w);
      }
#pragma unroll
      for (int r = 0; r < 2; r++)
#pragma unroll
        for (int t = 0; t < 2; t++)
          s[r][t] = fmaf(a[r].x, x[t].x, fmaf(a[r].y, x[t].y, fmaf(a[r].z, x[t].z, fmaf(a[r].w, x[t].w, s[r][t]))));
    }
#pragma unroll
    for (int r = 0; r < 2; r++) {
      bias[r] += sb[r];
#pragma unroll
      for (int t = 0; t < 2; t++) acc[r][t] += s[r][t];
    }
  }
#pragma unroll
  for (int r = 0; r < 2; r++) {
    const int o = ob + 16 * r;
    if (o >= Cout) continue;
#pragma unroll
    for (int t = 0; t < 2; t++)
      if (ib + 16 * t < Cin) atomicAdd(dW + o * Cin + ib + 16 * t, acc[r][t]);
    if (db && ib == 0) atomicAdd(db + o, bias[r]);
  }
}

// gelu in the tanh form, (1 + tanh u)/2 as the logistic function of 2u: no
// cancellation at negative u, and one exponential and one division instead
// of tanhf's two branches (it was a third of the inverse transform's time).
__device__ __forceinline__ float gelu_t(float z, float* dgdz) {
  const float k0 = 0.7978845608028654f, k1 = 0.044715f;
  const float u = k0 * (z + k1 * z * z * z);
  const float t = expf(-2.f * u), s = 1.f / (1.f + t);  // t = inf: s = 0
  if (dgdz) *dgdz = s + z * (fminf(t, 3e38f) * s * s) * (2.f * k0) * (1.f + 3.f * k1 * z * z);
  return z * s;
}

#include "fno_dft.cuh"

// t[c][k] = sum_j R[k][j][c] s[j][k] (complex, bf16 weights); one warp per
// mode k, lane c (C <= 32): the weight loads are coalesced, s is broadcast.
__global__ void k_mix_fwd(const float2* __restrict__ s, const uint16_t* __restrict__ R, float2* __restrict__ t,
                          int C, int K) {
  const int lane = threadIdx.x & 31;
  const int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (k >= K) return;
  float2 acc = make_float2(0.f, 0.f);
  if (lane < C) {
    const uint32_t* R2 = reinterpret_cast<const uint32_t*>(R);
#pragma unroll 8
    for (int j = 0; j < C; j++) {
      const uint32_t wbits = __ldcs(R2 + ((int64_t)k * C + j) * C + lane);  // read once per forward
      const float wr = __uint_as_float(wbits << 16), wi = __uint_as_float(wbits & 0xffff0000u);
      const float2 sj = s[(int64_t)j * K + k];
      acc.x = fmaf(wr, sj.x, fmaf(-wi, sj.y, acc.x));
      acc.y = fmaf(wr, sj.y, fmaf(wi, sj.x, acc.y));
    }
    t[(int64_t)lane * K + k] = acc;
  }
}

// Backward of the mixing, G_t scaled by a(kx)/V first (one warp per mode,
// lane c): dR[k][j][c] += conj(s[j][k]) g[c][k];
// gs[j][k] = sum_c conj(R[k][j][c]) g[c][k] (a warp reduction over c).
__global__ void k_mix_bwd(const float2* __restrict__ gt, const float2* __restrict__ s,
                          const uint16_t* __restrict__ R, float2* __restrict__ gs, float* __restrict__ dR, int C,
                          int K, int M, float invV) {
  const int lane = threadIdx.x & 31;
  const int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (k >= K) return;
  const float a = ((k % M) == 0 ? 1.f : 2.f) * invV;
  float2 g = make_float2(0.f, 0.f);
  if (lane < C) {
    g = gt[(int64_t)lane * K + k];
    g.x *= a;
    g.y *= a;
  }
  const uint32_t* R2 = reinterpret_cast<const uint32_t*>(R);
  float2* dR2 = reinterpret_cast<float2*>(dR);
  for (int j = 0; j < C; j++) {
    const float2 sj = s[(int64_t)j * K + k];
    float px = 0.f, py = 0.f;
    if (lane < C) {
      const int64_t r = ((int64_t)k * C + j) * C + lane;
      const uint32_t wbits = R2[r];
      const float wr = __uint_as_float(wbits << 16), wi = __uint_as_float(wbits & 0xffff0000u);
      px = wr * g.x + wi * g.y;  // conj(w) g
      py = wr * g.y - wi * g.x;
      float2 d = dR2[r];
      d.x += sj.x * g.x + sj.y * g.y;  // conj(s) g
      d.y += sj.x * g.y - sj.y * g.x;
      dR2[r] = d;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      px += __shfl_xor_sync(0xffffffffu, px, o);
      py += __shfl_xor_sync(0xffffffffu, py, o);
    }
    if (lane == 0) gs[(int64_t)j * K + k] = make_float2(px, py);
  }
}

// The same two for 32 channels, bound by the read of R (and of dR and its
// write): a CTA takes eight modes, a warp one of them, its 1024 weights in
// eight loads of 16 bytes a lane (lane: channels c = 4 (lane % 8) .., j =
// 4 jj + lane / 8), all requested before the spectra arrive; the spectra pass
// through shared memory, as eight modes are the 64 bytes that a channel keeps
// together. A lane per channel with 4-byte loads and 8-byte strided spectra:
// 17.8 us forward, 74 us backward at M = 16 (67 and 335 MB); now 13.2 us
// and 56 us (6.0 TB/s).
constexpr int MK = 8;   // modes per CTA
constexpr int MP = 34;  // pitch of a mode's channels: eight modes and two channels in distinct banks
__device__ __forceinline__ float2 wr_wi(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
__device__ __forceinline__ void load_modes(float2 (*s)[MP], const float2* __restrict__ in, int k0, int K) {
  const int m = threadIdx.x % MK, j = threadIdx.x / MK;
  s[m][j] = k0 + m < K ? *(in + (int64_t)j * K + k0 + m) : make_float2(0.f, 0.f);
}
__device__ __forceinline__ void store_modes(const float2 (*s)[MP], float2* __restrict__ out, int k0, int K) {
  const int m = threadIdx.x % MK, j = threadIdx.x / MK;
  if (k0 + m < K) out[(int64_t)j * K + k0 + m] = s[m][j];
}
__global__ void __launch_bounds__(256) k_mix_fwd32(const float2* __restrict__ s, const uint4* __restrict__ R,
                                                   float2* __restrict__ t, int K) {
  kernel_wait();
  s = after_wait(s);
  R = after_wait(R);
  __shared__ float2 sS[MK][MP], sO[MK][MP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, k0 = blockIdx.x * MK, k = k0 + warp;
  uint4 w[8];
#pragma unroll
  for (int jj = 0; jj < 8; jj++) w[jj] = k < K ? __ldcs(R + (int64_t)k * 256 + 32 * jj + lane) : make_uint4(0, 0, 0, 0);
  load_modes(sS, s, k0, K);
  __syncthreads();
  float2 acc[4];
#pragma unroll
  for (int c = 0; c < 4; c++) acc[c] = make_float2(0.f, 0.f);
#pragma unroll
  for (int jj = 0; jj < 8; jj++) {
    const float2 x = sS[warp][4 * jj + (lane >> 3)];
    const uint32_t u[4] = {w[jj].x, w[jj].y, w[jj].z, w[jj].w};
#pragma unroll
    for (int c = 0; c < 4; c++) {
      const float2 r = wr_wi(u[c]);
      acc[c].x = fmaf(r.x, x.x, fmaf(-r.y, x.y, acc[c].x));
      acc[c].y = fmaf(r.x, x.y, fmaf(r.y, x.x, acc[c].y));
    }
  }
#pragma unroll
  for (int o = 8; o < 32; o <<= 1)
#pragma unroll
    for (int c = 0; c < 4; c++) {
      acc[c].x += __shfl_xor_sync(0xffffffffu, acc[c].x, o);
      acc[c].y += __shfl_xor_sync(0xffffffffu, acc[c].y, o);
    }
  if (lane < 8) {
#pragma unroll
    for (int c = 0; c < 4; c++) sO[warp][4 * lane + c] = acc[c];
  }
  __syncthreads();
  store_modes(sO, t, k0, K);
}
__global__ void __launch_bounds__(256) k_mix_bwd32(const float2* __restrict__ gt, const float2* __restrict__ s,
                                                   const uint4* __restrict__ R, float2* __restrict__ gs,
                                                   float4* __restrict__ dR, int K, int M, float invV) {
  kernel_wait();
  gt = after_wait(gt);
  s = after_wait(s);
  R = after_wait(R);
  dR = after_wait(dR);
  __shared__ float2 sG[MK][MP], sS[MK][MP], sO[MK][MP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, k0 = blockIdx.x * MK, k = k0 + warp;
  const bool live = k < K;
  const int64_t base = (int64_t)k * 256 + lane;
  uint4 w[8];  // before any store: they are not moved past one
#pragma unroll
  for (int jj = 0; jj < 8; jj++) w[jj] = live ? __ldcs(R + base + 32 * jj) : make_uint4(0, 0, 0, 0);
  load_modes(sG, gt, k0, K);
  load_modes(sS, s, k0, K);
  __syncthreads();
  const float a = ((k % M) == 0 ? 1.f : 2.f) * invV;
  float2 g[4], p[8];
#pragma unroll
  for (int c = 0; c < 4; c++) {
    g[c] = sG[warp][4 * (lane & 7) + c];
    g[c].x *= a;
    g[c].y *= a;
  }
#pragma unroll
  for (int half = 0; half < 2; half++) {
    float4 d[4][2];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int64_t r = base + 32 * (4 * half + q);
      d[q][0] = live ? __ldcs(dR + 2 * r) : make_float4(0.f, 0.f, 0.f, 0.f);
      d[q][1] = live ? __ldcs(dR + 2 * r + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int jj = 4 * half + q;
      const float2 x = sS[warp][4 * jj + (lane >> 3)];
      const uint32_t u[4] = {w[jj].x, w[jj].y, w[jj].z, w[jj].w};
      p[jj] = make_float2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < 4; c++) {
        const float2 r = wr_wi(u[c]);
        p[jj].x = fmaf(r.x, g[c].x, fmaf(r.y, g[c].y, p[jj].x));  // conj(w) g
        p[jj].y = fmaf(r.x, g[c].y, fmaf(-r.y, g[c].x, p[jj].y));
        float4& v = d[q][c >> 1];
        float& vx = (c & 1) ? v.z : v.x;
        float& vy = (c & 1) ? v.w : v.y;
        vx += x.x * g[c].x + x.y * g[c].y;  // conj(s) g
        vy += x.x * g[c].y - x.y * g[c].x;
      }
      if (live) {
        const int64_t r = base + 32 * jj;
        __stcs(dR + 2 * r, d[q][0]);
        __stcs(dR + 2 * r + 1, d[q][1]);
      }
    }
  }
  // sums over the 8 lanes of a j: each step halves the j's a lane keeps
#pragma unroll
  for (int h = 4; h > 0; h >>= 1) {
    const bool up = lane & h;
#pragma unroll
    for (int q = 0; q < h; q++) {
      const float2 keep = up ? p[q + h] : p[q], send = up ? p[q] : p[q + h];
      p[q].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, h);
      p[q].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, h);
    }
  }
  sO[warp][4 * (lane & 7) + (lane >> 3)] = p[0];
  __syncthreads();
  store_modes(sO, gs, k0, K);
}
// 32 channels, and weights on 16-byte boundaries
bool mix32(int C, const void* R, const void* dR) {
  return C == 32 && ((reinterpret_cast<uintptr_t>(R) | reinterpret_cast<uintptr_t>(dR)) & 15) == 0;
}

__global__ void __launch_bounds__(256) k_gelu_bwd(const float4* __restrict__ z, const float4* __restrict__ dv,
                                                  float4* __restrict__ dz, int64_t n4) {
  kernel_wait();
  z = after_wait(z);
  dv = after_wait(dv);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 a = *(z + i), b = *(dv + i);
    float4 d;
    gelu_t(a.x, &d.x);
    gelu_t(a.y, &d.y);
    gelu_t(a.z, &d.z);
    gelu_t(a.w, &d.w);
    dz[i] = make_float4(b.x * d.x, b.y * d.y, b.z * d.z, b.w * d.w);
  }
}

// Sum over the CTA (of 256 threads) of r, added to out by its first thread.
__device__ __forceinline__ void block_add(double r, double* out) {
  __shared__ double part[8];
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = r;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) r += part[w];
    atomicAdd(out, r);
  }
}

// Sum of the squares in FP64, added to out: few floats, or a misaligned array.
__global__ void __launch_bounds__(256) k_sumsq(const float* t, int64_t n, double* out) {
  kernel_wait();
  t = after_wait(t);
  double r = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    r += (double)t[i] * t[i];
  block_add(r, out);
}

__global__ void k_loss(const float* y, const float* t, float* dy, int64_t n, const double* tnorm, float weight,
                       double* loss) {
  kernel_wait();
  y = after_wait(y);
  t = after_wait(t);
  tnorm = after_wait(tnorm);
  __shared__ double s_inv;
  if (threadIdx.x == 0) s_inv = 1.0 / fmax(*tnorm, 1e-300);
  __syncthreads();
  const double inv = s_inv;
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float d = y[i] - t[i];
    s += (double)d * d;
    dy[i] = (float)(2.0 * d * inv) * weight;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, s * inv * weight);
}

// The same of many floats (16-byte aligned). Bound by the read: every product is
// exact as two floats and the sums are compensated (FP32 pairs, about 48 bits),
// as this GPU's FP64 rate is a 64th of its FP32 rate. A thread whose values
// leave the range where that is exact enough (past 1e18 in size, all below
// 1e-12, infinities, NaNs) sums them in FP64. Over many threads the pairs'
// roundings average out: against the exact sum 1e-15 (rms) for 98304 floats and
// 1.2e-15 for 5e6, where FP64 sums with an unordered add per warp are off by
// 1.5e-15 and 6.5e-15. For few they do not (1.5e-15 against 2e-16 for 64
// floats): below PAIRS floats the sum is k_sumsq's. 134e6 floats: 252 us (FP64
// sums) -> 96 us, 5.6 TB/s; 786432 floats: 40 -> 6 us.
constexpr int64_t PAIRS = 65536;
__global__ void __launch_bounds__(256) k_gradnorm(const float4* __restrict__ t, int64_t n4, const float* __restrict__ tail,
                                                  int ntail, double* out) {
  kernel_wait();
  t = after_wait(t);
  tail = after_wait(tail);
  float s[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f}, top = 0.f;
  auto add = [&](int k, float x) {
    const float p = __fmul_rn(x, x), e = __fmaf_rn(x, x, -p);
    const float u = __fadd_rn(s[k], p), d = __fsub_rn(u, s[k]);
    c[k] += __fadd_rn(__fadd_rn(__fsub_rn(s[k], __fsub_rn(u, d)), __fsub_rn(p, d)), e);
    s[k] = u;
    top = fmaxf(top, fabsf(x));
  };
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
#pragma unroll 4
  for (int64_t i = i0; i < n4; i += stride) {
    const float4 x = *(t + i);
    add(0, x.x);
    add(1, x.y);
    add(2, x.z);
    add(3, x.w);
  }
  if (i0 < ntail) add(0, tail[i0]);
  double r = 0.0;
  const float sum = (s[0] + s[1]) + (s[2] + s[3]);
  if (isfinite(sum) && top < 1e18f && (top == 0.f || top > 1e-12f)) {
    // the four sums as one float pair, then one FP64 addition a thread
#pragma unroll
    for (int k = 1; k < 4; k++) {
      const float u = __fadd_rn(s[0], s[k]), d = __fsub_rn(u, s[0]);
      c[0] += __fadd_rn(__fadd_rn(__fsub_rn(s[0], __fsub_rn(u, d)), __fsub_rn(s[k], d)), c[k]);
      s[0] = u;
    }
    r = (double)s[0] + (double)c[0];
  } else {
    for (int64_t i = i0; i < n4; i += stride) {
      const float4 x = *(t + i);
      r += (double)x.x * x.x + (double)x.y * x.y + (double)x.z * x.z + (double)x.w * x.w;
    }
    if (i0 < ntail) r += (double)tail[i0] * tail[i0];
  }
  block_add(r, out);
}

struct AdamArgs {
  float lr, b1, b2, eps, c1, c2, clip;
  const double* sumsq;
};
// Scale of the gradient: clipped to the norm, negative when it is not finite.
__device__ __forceinline__ float adam_scale(const AdamArgs& a) {
  const double norm = sqrt(*a.sumsq);
  if (!isfinite(norm)) return -1.f;  // drop the step, keep parameters and moments
  return (a.clip > 0.f && norm > a.clip) ? (float)(a.clip / norm) : 1.f;
}
__device__ __forceinline__ void adam1(const AdamArgs& a, float scale, float& p, float g, float& m, float& v) {
  if (scale < 0.f) return;
  const float gi = g * scale;
  const float mi = a.b1 * m + (1.f - a.b1) * gi;
  const float vi = a.b2 * v + (1.f - a.b2) * gi * gi;
  m = mi;
  v = vi;
  p -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
}

// One Adam step; the bfloat16 copy of the parameters too when pb is not null.
// Bound by HBM: four arrays in, four and the copy out, 34 bytes a parameter;
// four parameters per thread and step. 134e6 parameters, with the copy: 1.25
// (two kernels) -> 0.68 ms, 6.7 TB/s.
__global__ void __launch_bounds__(256) k_adam(int64_t n, float* p, float* g, float* m, float* v, uint16_t* pb,
                                              AdamArgs a, int vec) {
  kernel_wait();
  p = after_wait(p);
  g = after_wait(g);
  m = after_wait(m);
  v = after_wait(v);
  a.sumsq = after_wait(a.sumsq);
  __shared__ float s_scale;  // one thread takes the FP64 square root
  if (threadIdx.x == 0) s_scale = adam_scale(a);
  __syncthreads();
  const float scale = s_scale;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n4 = vec ? n / 4 : 0;
#pragma unroll 2
  for (int64_t i = i0; i < n4; i += stride) {
    float4 P = __ldcs(reinterpret_cast<float4*>(p) + i), M = __ldcs(reinterpret_cast<float4*>(m) + i),
           V = __ldcs(reinterpret_cast<float4*>(v) + i);
    const float4 G = __ldcs(reinterpret_cast<float4*>(g) + i);
    adam1(a, scale, P.x, G.x, M.x, V.x);
    adam1(a, scale, P.y, G.y, M.y, V.y);
    adam1(a, scale, P.z, G.z, M.z, V.z);
    adam1(a, scale, P.w, G.w, M.w, V.w);
    __stcs(reinterpret_cast<float4*>(p) + i, P);
    __stcs(reinterpret_cast<float4*>(m) + i, M);
    __stcs(reinterpret_cast<float4*>(v) + i, V);
    __stcs(reinterpret_cast<float4*>(g) + i, make_float4(0.f, 0.f, 0.f, 0.f));
    if (pb) *reinterpret_cast<uint2*>(pb + 4 * i) = make_uint2(pack_bf16(P.x, P.y), pack_bf16(P.z, P.w));
  }
  for (int64_t i = 4 * n4 + i0; i < n; i += stride) {
    float P = p[i], M = m[i], V = v[i];
    adam1(a, scale, P, g[i], M, V);
    p[i] = P;
    m[i] = M;
    v[i] = V;
    g[i] = 0.f;
    if (pb) pb[i] = __bfloat16_as_ushort(__float2bfloat16_rn(P));
  }
}

__global__ void k_cast(const float* p, uint16_t* q, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    q[i] = __bfloat16_as_ushort(__float2bfloat16_rn(p[i]));
}

// splitmix64 hash -> uniform in [-1, 1)
__device__ __forceinline__ float hash_uniform(uint64_t seed, uint64_t i) {
  uint64_t z = seed + 0x9E3779B97F4A7C15ull * (i + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return (float)((double)(z >> 11) * (1.0 / 9007199254740992.0)) * 2.f - 1.f;
}

__global__ void k_init(Shape s, uint64_t seed, float* p) {
  const int64_t n = s.count();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float scale = 0.f;  // biases start at zero
    if (i < s.off_p()) scale = sqrtf(1.f / 4.f);
    else if (i >= s.off_Q() && i < s.off_q()) scale = sqrtf(1.f / s.C);
    else if (i >= s.off_layer(0) && i < s.off_Q()) {
      const int64_t r = (i - s.off_layer(0)) % s.layer_size();
      if (r < (int64_t)s.C * s.C) scale = sqrtf(1.f / s.C);
      else if (r >= (int64_t)s.C * s.C + s.C) scale = 1.f / ((float)s.C * s.C);
    }
    p[i] = scale * hash_uniform(seed, (uint64_t)i);
  }
}

// Block means over f^3 cells, one CTA per coarse row (c, z, y): threads run
// along the fine x axis summing the f x f fine rows (coalesced), then f
// neighbours are summed through shared memory.
__global__ void k_coarsen(int N, int n, const float* __restrict__ fine, const float* __restrict__ fine2,
                          float* __restrict__ coarse, const float* __restrict__ scale) {
  extern __shared__ float sx[];  // N floats
  const int f = N / n;
  const int row = blockIdx.x;  // (c n + z) n + y
  const int y = row % n, z = (row / n) % n, c = row / (n * n);
  const int64_t N3 = (int64_t)N * N * N;
  const float* src = fine + c * N3;
  const float* src2 = fine2 ? fine2 + c * N3 : nullptr;
  for (int x = threadIdx.x; x < N; x += blockDim.x) {
    float acc = 0.f;
    for (int dz = 0; dz < f; dz++)
      for (int dy = 0; dy < f; dy++) {
        const int64_t i = ((int64_t)(z * f + dz) * N + (y * f + dy)) * N + x;
        acc += src2 ? 0.5f * (src[i] + src2[i]) : src[i];
      }
    sx[x] = acc;
  }
  __syncthreads();
  const float d = (float)f * f * f * (scale ? *scale : 1.f);
  for (int xc = threadIdx.x; xc < n; xc += blockDim.x) {
    float acc = 0.f;
    for (int dx = 0; dx < f; dx++) acc += sx[xc * f + dx];
    coarse[(int64_t)row * n + xc] = acc / d;
  }
}

// The same with 16-byte loads, rows split over the CTA (N / 4 lanes along x,
// RY row groups), so that a thread has several loads in flight. Bound by the
// read: 256^3 -> 64^3, three components (201 MB): 55 us with 4-byte loads, now
// 49 us (4.1 TB/s).
__global__ void __launch_bounds__(256, 6) k_coarsen4(int N, int n, const float4* __restrict__ fine,
                                                  const float4* __restrict__ fine2, float* __restrict__ coarse,
                                                  const float* __restrict__ scale) {
  kernel_wait();
  fine = after_wait(fine);
  fine2 = after_wait(fine2);
  scale = after_wait(scale);
  extern __shared__ __align__(16) float sx[];  // [RY][N]
  const int f = N / n, TX = N / 4, RY = blockDim.y, xq = threadIdx.x, ry = threadIdx.y;
  const int row = (blockIdx.z * n + blockIdx.y) * n + blockIdx.x;
  const int y = blockIdx.x, z = blockIdx.y, c = blockIdx.z;
  const int64_t base = (((int64_t)c * N + z * f) * N + y * f) * TX + xq;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  int off = ry * TX, dy = ry;  // row dy of plane dz: at most f N TX = 2^28 (N <= 1024)
  while (dy >= f) dy -= f, off += (N - f) * TX;
#pragma unroll 4
  for (int r = ry; r < f * f; r += RY) {
    float4 v = __ldcs(fine + base + off);
    if (fine2) {
      const float4 u = __ldcs(fine2 + base + off);
      v = make_float4(0.5f * (v.x + u.x), 0.5f * (v.y + u.y), 0.5f * (v.z + u.z), 0.5f * (v.w + u.w));
    }
    acc = make_float4(acc.x + v.x, acc.y + v.y, acc.z + v.z, acc.w + v.w);
    dy += RY;
    off += RY * TX;
    while (dy >= f) dy -= f, off += (N - f) * TX;
  }
  const float d = (float)f * f * f * (scale ? *scale : 1.f);
  if (f % 4 == 0) {  // a quad lies in one coarse cell
    sx[ry * TX + xq] = (acc.x + acc.y) + (acc.z + acc.w);
    __syncthreads();
    for (int xc = ry * TX + xq; xc < n; xc += RY * TX) {
      float a = 0.f;
      for (int r = 0; r < RY; r++)
        for (int t = 0; t < f / 4; t++) a += sx[r * TX + xc * (f / 4) + t];
      coarse[(int64_t)row * n + xc] = a / d;
    }
    return;
  }
  *reinterpret_cast<float4*>(sx + ry * N + 4 * xq) = acc;
  __syncthreads();
  for (int xc = ry * TX + xq; xc < n; xc += RY * TX) {
    float a = 0.f;
    for (int r = 0; r < RY; r++)
      for (int dx = 0; dx < f; dx++) a += sx[r * N + xc * f + dx];
    coarse[(int64_t)row * n + xc] = a / d;
  }
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

void launch_coarsen(int N, int n, int ncomp, const float* fine, const float* fine2, float* coarse,
                    const float* scale, cudaStream_t st) {
  if (N % 4 == 0 && N <= 1024 && ncomp < 65536 && aligned16(fine) && aligned16(fine2)) {
    const int f = N / n, TX = N / 4, RY = std::min(f * f, 256 / TX);
    launch_early(k_coarsen4, dim3(n, n, ncomp), dim3(TX, RY), sizeof(float) * N * RY, st, N, n,
                 reinterpret_cast<const float4*>(fine), reinterpret_cast<const float4*>(fine2), coarse, scale);
    return;
  }
  const int threads = N < 256 ? ((N + 31) / 32) * 32 : 256;
  k_coarsen<<<(unsigned)(ncomp * n * n), threads, sizeof(float) * N, st>>>(N, n, fine, fine2, coarse, scale);
}

__global__ void k_input(int n, float a0, const float* g, const double* sumsq, float* x, float* scale_out) {
  kernel_wait();
  g = after_wait(g);
  sumsq = after_wait(sumsq);
  const int64_t V = (int64_t)n * n * n;
  __shared__ float s_rms;  // one thread a CTA does the FP64 arithmetic
  if (threadIdx.x == 0) s_rms = (float)sqrt(fmax(*sumsq / (3.0 * V), 1e-60));
  __syncthreads();
  const float s = s_rms;
  if (blockIdx.x == 0 && threadIdx.x == 0) *scale_out = s;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
    const float gx = g[v], gy = g[V + v], gz = g[2 * V + v];
    x[v] = gx / s;
    x[V + v] = gy / s;
    x[2 * V + v] = gz / s;
    x[3 * V + v] = 0.25f * log10f(sqrtf(gx * gx + gy * gy + gz * gz) / a0 + 1e-12f);
  }
}

// Cubic convolution weights (Keys, a = -1/2) of the taps -1, 0, 1, 2 at
// fraction u in [0, 1).
__device__ __forceinline__ void cubic_w(float u, float w[4]) {
  w[0] = ((-u + 2.f) * u - 1.f) * u * 0.5f;
  w[1] = ((3.f * u - 5.f) * u * u + 2.f) * 0.5f;
  w[2] = ((-3.f * u + 4.f) * u + 1.f) * u * 0.5f;
  w[3] = (u - 1.f) * u * u * 0.5f;
}

// Periodic cubic-convolution upsampling, one axis per kernel: the fine cell
// centre X of the fine axis (f = N/n fine cells per coarse cell) sits at
// coarse position (X + 1/2)/f - 1/2; the taps are the coarse cells x0 - 1 ..
// x0 + 2 around it. Each kernel reads `in` with the axis of length n at
// stride `stride` (elements) inside rows of `inner` elements, and writes the
// axis of length N. One CTA per outer row; threads along the inner axis.
__device__ __forceinline__ void up_taps(int X, int n, int f, int idx[4], float w[4]) {
  const float fx = (X + 0.5f) / f - 0.5f;
  const int x0 = (int)floorf(fx);
  cubic_w(fx - x0, w);
#pragma unroll
  for (int k = 0; k < 4; k++) idx[k] = ((x0 - 1 + k) % n + n) % n;
}

// x: in [rows][n] -> out [rows][N]
__global__ void k_up_x(int n, int N, const float* __restrict__ in, float* __restrict__ out) {
  const int f = N / n;
  const int64_t row = blockIdx.x;
  for (int X = threadIdx.x; X < N; X += blockDim.x) {
    int idx[4];
    float w[4];
    up_taps(X, n, f, idx, w);
    const float* r = in + row * n;
    out[row * N + X] = w[0] * r[idx[0]] + w[1] * r[idx[1]] + w[2] * r[idx[2]] + w[3] * r[idx[3]];
  }
}

// One axis of the upsampling, in [outer][n][inner] -> out [outer][N][inner]
// (times scale when given), by coarse interval: CTA row (outer, j) reads the
// four coarse rows j-1..j+2 once per inner index and writes the f = N / n fine
// rows whose taps they are, Y = f j + f/2 + q (mod N), q < f (the fine rows
// with floor((Y + 1/2)/f - 1/2) = j). blockIdx.y splits the inner axis.
__global__ void k_up_axis(int n, int N, int64_t inner, int64_t chunk, const float* __restrict__ in,
                          float* __restrict__ out, const float* __restrict__ scale) {
  extern __shared__ float upw[];  // f x 4 weights
  __shared__ int upy[64];         // fine row of each q (f <= 64)
  const int f = N / n;
  const int j = (int)(blockIdx.x % n);
  const int64_t outer = blockIdx.x / n;
  for (int q = threadIdx.x; q < f; q += blockDim.x) {
    const int Y = (f * j + f / 2 + q) % N;
    int idx[4];
    up_taps(Y, n, f, idx, upw + 4 * q);
    upy[q] = Y;
  }
  __syncthreads();
  const float s = scale ? *scale : 1.f;
  const float* b0 = in + (outer * n + (j - 1 + n) % n) * inner;
  const float* b1 = in + (outer * n + j) * inner;
  const float* b2 = in + (outer * n + (j + 1) % n) * inner;
  const float* b3 = in + (outer * n + (j + 2) % n) * inner;
  float* o = out + outer * N * inner;
  const int64_t x0 = (int64_t)blockIdx.y * chunk, x1 = min(inner, x0 + chunk);
  for (int64_t X = x0 + threadIdx.x; X < x1; X += blockDim.x) {
    const float v0 = __ldg(b0 + X), v1 = __ldg(b1 + X), v2 = __ldg(b2 + X), v3 = __ldg(b3 + X);
    for (int q = 0; q < f; q++) {
      const float* w = upw + 4 * q;
      const float v = w[0] * v0 + w[1] * v1 + w[2] * v2 + w[3] * v3;
      o[(int64_t)upy[q] * inner + X] = s * v;
    }
  }
}

// All three axes in one pass, for factors f = N/n and coarse sides n that are
// multiples of four: a CTA takes one coarse interval along y and UPZ of them
// along z in turn (four of the f fine planes of each: blockIdx.z), interpolates
// the coarse rows along y, then z (in shared memory, on the coarse x), and
// writes 4 f fine rows, a thread always the same four neighbouring x. Bound by the write; the
// three passes it replaces also wrote and read the two steps between: 64^3 ->
// 256^3, three components (201 MB): 120 us, now 54 us
// (3.8 TB/s; its instructions take 80% of the issue slots). Other factors and
// sides keep the three passes.
constexpr int UPZ = 4;
size_t smem_up3(int n, int N) { return sizeof(float) * (16 * (size_t)n + 8 * (size_t)N + 4 * (size_t)(N / n)); }
__global__ void __launch_bounds__(256) k_up3(int n, int N, const float4* __restrict__ in, float4* __restrict__ out,
                                             const float* __restrict__ scale) {
  extern __shared__ __align__(16) float sm[];
  const int f = N / n, n4 = n / 4, TX = N / 4, RY = blockDim.y;  // TX float4s: a fine row, or f coarse rows
  const int xq = threadIdx.x, ry = threadIdx.y, q = xq / n4, i4 = xq - q * n4;
  float4* sC = reinterpret_cast<float4*>(sm);  // [4 z][4 y][n], coarse
  float4* sP = sC + 16 * n4;                   // [4 z][f][n], fine along y
  float4* sQ = sP + 4 * TX;                    // [4][f][n], fine along z too
  float4* sw = sQ + 4 * TX;                    // [f] weights of the fine positions of an interval
  const int jy = blockIdx.x, jz0 = UPZ * blockIdx.y, c = blockIdx.z % 3, q0 = 4 * (blockIdx.z / 3);
  auto wrap = [](int i, int m) { return i < 0 ? i + m : i < m ? i : i - m; };
  for (int p = ry * TX + xq; p < f; p += RY * TX) {
    float w[4];
    cubic_w((f / 2 + p + 0.5f) / f - 0.5f, w);  // f j + f/2 + p is that far past the coarse position j
    sw[p] = make_float4(w[0], w[1], w[2], w[3]);
  }
  __syncthreads();
  auto mix = [](float4 w, float4 a, float4 b, float4 d, float4 e, float s) {
    return make_float4(s * (w.x * a.x + w.y * b.x + w.z * d.x + w.w * e.x),
                       s * (w.x * a.y + w.y * b.y + w.z * d.y + w.w * e.y),
                       s * (w.x * a.z + w.y * b.z + w.z * d.z + w.w * e.z),
                       s * (w.x * a.w + w.y * b.w + w.z * d.w + w.w * e.w));
  };
  kernel_wait();
  in = after_wait(in);
  scale = after_wait(scale);
  // x: weights and coarse cells of this thread's four positions X0 + k of the
  // coarse cell i, which lie past the coarse position i - 1 or, from f/2 on, i
  const float s = *scale;
  const int X0 = 4 * xq, i = X0 / f, x0 = X0 - i * f, h = f / 2;
  float4 wx[4];
#pragma unroll
  for (int k = 0; k < 4; k++) wx[k] = sw[x0 + k < h ? x0 + k + h : x0 + k - h];
  const int first = i - (x0 < h ? 2 : 1);
  const bool far = x0 < h && x0 + 2 >= h;  // the taps move on by a cell between X0 + 1 and X0 + 2 (h is even)
  int idx[5];
#pragma unroll
  for (int k = 0; k < 5; k++) idx[k] = wrap(first + k, n);
  const int Y0 = f * jy + h;
  for (int step = 0; step < UPZ; step++) {
    // coarse plane jz - 1 + k is in slot (step + k) % 4 of sC and sP
    const int jz = jz0 + step, k0 = step ? 3 : 0;
    for (int r = 4 * k0 + ry * f + q; r < 16; r += RY * f) {
      const int z = wrap(jz - 1 + r / 4, n), y = wrap(jy - 1 + r % 4, n);
      sC[(4 * ((step + r / 4) & 3) + r % 4) * n4 + i4] = *(in + (((int64_t)c * n + z) * n + y) * n4 + i4);
    }
    __syncthreads();
    for (int k = k0 + ry; k < 4; k += RY) {
      const int slot = (step + k) & 3;
      const float4* v = sC + 4 * slot * n4 + i4;
      sP[slot * TX + xq] = mix(sw[q], v[0], v[n4], v[2 * n4], v[3 * n4], 1.f);
    }
    __syncthreads();
    {
      const float4 a = sP[(step & 3) * TX + xq], b = sP[((step + 1) & 3) * TX + xq],
                   d = sP[((step + 2) & 3) * TX + xq], e = sP[((step + 3) & 3) * TX + xq];
      for (int z = ry; z < 4; z += RY) sQ[z * TX + xq] = mix(sw[q0 + z], a, b, d, e, s);
    }
    __syncthreads();
    const int Z0 = f * jz + h + q0;
    int qz = 0, qy = ry;  // fine row: plane Z0 + qz, row Y0 + qy of the interval
    for (;; qy += RY) {
      while (qy >= f) qy -= f, qz++;
      if (qz >= 4) break;
      const float* v = reinterpret_cast<const float*>(sQ) + (qz * f + qy) * n;
      const float a = v[idx[0]], b = v[idx[1]], d = v[idx[2]], e = v[idx[3]], g = v[idx[4]];
      const float a2 = far ? b : a, b2 = far ? d : b, d2 = far ? e : d, e2 = far ? g : e;
      float4 o;
      o.x = wx[0].x * a + wx[0].y * b + wx[0].z * d + wx[0].w * e;
      o.y = wx[1].x * a + wx[1].y * b + wx[1].z * d + wx[1].w * e;
      o.z = wx[2].x * a2 + wx[2].y * b2 + wx[2].z * d2 + wx[2].w * e2;
      o.w = wx[3].x * a2 + wx[3].y * b2 + wx[3].z * d2 + wx[3].w * e2;
      __stcs(out + (((int64_t)c * N + wrap(Z0 + qz, N)) * N + wrap(Y0 + qy, N)) * TX + xq, o);
    }
  }
}

// Sphere mixture on the mesh (Plummer: 3M/(4 pi a^3) (1 + r^2/a^2)^{-5/2};
// Hernquist: M a / (2 pi r (r + a)^3) with r >= 1/2 px), truncated at rmax.
__global__ void k_mixture(int N, float s, int K, const float* centre, const float* mass, const float* radius,
                          const int* kind, float rmax, float* rho) {
  const int64_t NF = (int64_t)N * N * N;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < NF; v += (int64_t)gridDim.x * blockDim.x) {
    const float X = (float)(v % N) - N / 2, Y = (float)((v / N) % N) - N / 2, Z = (float)(v / ((int64_t)N * N)) - N / 2;
    float acc = 0.f;
    for (int j = 0; j < K; j++) {
      const float dx = X - centre[3 * j], dy = Y - centre[3 * j + 1], dz = Z - centre[3 * j + 2];
      float r = sqrtf(dx * dx + dy * dy + dz * dz);
      if (r > rmax) continue;
      const float a = radius[j], m = mass[j];
      if (kind[j] == 0) {
        const float q = 1.f + r * r / (a * a);
        acc += 3.f * m / (4.f * 3.14159265358979f * a * a * a) * powf(q, -2.5f);
      } else {
        r = fmaxf(r, 0.5f);
        acc += m * a / (2.f * 3.14159265358979f * r * (r + a) * (r + a) * (r + a));
      }
    }
    rho[v] = acc / (s * s * s);
  }
}

unsigned grid_stride(int64_t n) {
  int64_t b = (n + TB - 1) / TB;
  return (unsigned)(b < 4096 ? b : 4096);
}

// *out += the sum of the squares of t.
void sumsq(const float* t, int64_t n, double* out, cudaStream_t st) {
  if (aligned16(t) && n >= PAIRS)
    // eight vectors a thread at least: a thread ends with FP64 sums
    launch_early(k_gradnorm, grid_stride((n + 31) / 32), TB, 0, st, reinterpret_cast<const float4*>(t), n / 4,
                 t + n / 4 * 4, (int)(n % 4), out);
  else
    launch_early(k_sumsq, grid_stride((n + 3) / 4), TB, 0, st, t, n, out);
}

// The plane kernels may need more than the default 48 KB of shared memory.
template <typename K>
bool opt_in(K kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024) == cudaSuccess;
}
template <int NX, int MX, bool FULL = false>
bool opt_in_xy() {
  return opt_in(dft::k_xy_fwd<NX, MX, FULL>) && opt_in(dft::k_xy_inv<NX, MX, FULL>);
}
bool smem_opt_in() {
  static const bool ok = opt_in_xy<16, 8>() && opt_in_xy<32, 8>() && opt_in_xy<32, 16>() && opt_in_xy<64, 8>() &&
                         opt_in_xy<64, 16>() && opt_in_xy<64, 32>() && opt_in_xy<16, 8, true>() &&
                         opt_in_xy<32, 16, true>() && opt_in_xy<64, 16, true>();
  return ok;
}
// Calls f(NX, MX, FULL) with the transform kernels' bounds on n and M. FULL: the
// sides of the default networks, a training step 3.11 -> 1.56 ms at 32 (with the
// unfolded sums before); the sides between the bounds gain as much from the
// folding: 1.50 -> 0.73 ms at 24, 3.52 -> 1.82 at 40, 3.69 -> 1.82 at 48, 4.14 ->
// 1.99 at 56.
template <typename F>
void by_size(int n, int M, F f) {
  std::integral_constant<int, 8> c8;
  std::integral_constant<int, 16> c16;
  std::integral_constant<int, 32> c32;
  std::integral_constant<int, 64> c64;
  std::true_type full;
  std::false_type part;
  if (n == 16 && M == 8) f(c16, c8, full);
  else if (n == 32 && M == 16) f(c32, c16, full);
  else if (n == 64 && M == 16) f(c64, c16, full);
  else if (n <= 16) f(c16, c8, part);
  else if (n <= 32) M <= 8 ? f(c32, c8, part) : f(c32, c16, part);
  else if (M <= 8) f(c64, c8, part);
  else M <= 16 ? f(c64, c16, part) : f(c64, c32, part);
}
// Plane kernels: two persistent CTAs per SM, each streaming its planes.
unsigned plane_grid(int planes) { return (unsigned)std::min(planes, 2 * 152); }

// Forward transform of C channels of real fields v -> out [C][K] (kept modes).
void dft3(const Shape& s, const Work& w, const float* v, float2* out, cudaStream_t st) {
  const int n = s.n, M = s.M, C = s.C, Iz = 2 * M * M, np = C * n;
  const size_t sz = dft::smem_z(n, M, n / 2, n / 2);
  const dim3 gz((Iz + dft::ZC - 1) / dft::ZC, C);
  by_size(n, M, [&](auto nx, auto mx, auto full) {
    constexpr int NX = nx.value, MX = mx.value;
    constexpr bool FULL = full.value;
    launch_early(dft::k_xy_fwd<NX, MX, FULL>, plane_grid(np), dft::TH, dft::smem_xy_fwd(n, M), st, v, w.b, n, M, np);
    launch_early(dft::k_z_fwd<NX, MX, FULL>, gz, dft::TH, sz, st, w.b, out, n, M, Iz);
  });
}

// Inverse transform of [C][K] kept modes, added into z; act as in k_xy_inv.
// adjoint: without the weights a(kx)/V, the adjoint of the forward transform.
void idft3(const Shape& s, const Work& w, const float2* in, float* z, float* v, bool adjoint, int act,
           cudaStream_t st) {
  const int n = s.n, M = s.M, C = s.C, Iz = 2 * M * M, np = C * n;
  const float w0 = adjoint ? 1.f : 1.f / (float)s.V, w1 = adjoint ? 1.f : 2.f * w0;
  const size_t sz = dft::smem_z(n, M, M + 1, n / 2 + 1);
  const dim3 gz((Iz + dft::ZC - 1) / dft::ZC, C);
  by_size(n, M, [&](auto nx, auto mx, auto full) {
    constexpr int NX = nx.value, MX = mx.value;
    constexpr bool FULL = full.value;
    launch_early(dft::k_z_inv<NX, MX, FULL>, gz, dft::TH, sz, st, in, w.b, n, M, Iz);
    launch_early(dft::k_xy_inv<NX, MX, FULL>, plane_grid(np), dft::TH, dft::smem_xy_inv(n, M), st, w.b, z, v, n, M,
                 w0, w1, act, np);
  });
}

void pw(const float* in, int Cin, const uint16_t* W, const uint16_t* b, int Cout, float* out, int64_t V,
        int transpose, cudaStream_t st) {
  const unsigned g = grid_stride(V);
  if (Cin <= 4) {
    launch_early(k_pw<4>, g, TB, 0, st, in, Cin, W, b, Cout, out, V, transpose);
  } else {
    // tensor cores: one warp per 32 voxels a step (V = n^3 is a multiple of 64), two CTAs per SM
    const unsigned gm = (unsigned)std::min<int64_t>((V / 32 + 7) / 8, 152 * 2);
    const int vec = aligned16(out);
    if (Cout <= 16) launch_early(k_pw_mma<1>, gm, TB, 0, st, in, Cin, W, b, Cout, out, V, transpose, vec);
    else launch_early(k_pw_mma<2>, gm, TB, 0, st, in, Cin, W, b, Cout, out, V, transpose, vec);
  }
}

}  // namespace

extern "C" {

int mond_fno_param_count(mond_fno_shape sh, int64_t* count) {
  Shape s;
  if (!count || !make_shape(sh, &s)) return -1;
  *count = s.count();
  return 0;
}

int mond_fno_workspace_bytes(mond_fno_shape sh, size_t* bytes) {
  Shape s;
  if (!bytes || !make_shape(sh, &s)) return -1;
  *bytes = carve(s, nullptr, nullptr);
  return 0;
}

int mond_fno_init(mond_fno_shape sh, uint64_t seed, float* params, void* stream) {
  Shape s;
  if (!params || !make_shape(sh, &s)) return -1;
  k_init<<<grid_stride(s.count()), TB, 0, (cudaStream_t)stream>>>(s, seed, params);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int mond_fno_cast(mond_fno_shape sh, const float* params, uint16_t* pb, void* stream) {
  Shape s;
  if (!params || !pb || !make_shape(sh, &s)) return -1;
  k_cast<<<grid_stride(s.count()), TB, 0, (cudaStream_t)stream>>>(params, pb, s.count());
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int mond_fno_forward(mond_fno_shape sh, const uint16_t* P, const float* x, float* y, void* workspace, void* stream) {
  Shape s;
  if (!P || !x || !y || !workspace || !make_shape(sh, &s)) return -1;
  cudaStream_t st = (cudaStream_t)stream;
  if (!smem_opt_in()) return -3;
  Work w;
  carve(s, (char*)workspace, &w);
  const int C = s.C;
  const int64_t V = s.V, CV = (int64_t)C * V;
  const unsigned warps_grid = (unsigned)(((int64_t)s.K * 32 + TB - 1) / TB);
  pw(x, 4, P + s.off_P(), P + s.off_p(), C, w.v, V, 0, st);
  for (int l = 0; l < s.L; l++) {
    const float* vl = w.v + l * CV;
    float* zl = w.z + l * CV;
    float2* shat = w.shat + (int64_t)l * C * s.K;
    pw(vl, C, P + s.off_W(l), P + s.off_b(l), C, zl, V, 0, st);
    dft3(s, w, vl, shat, st);
    const uint16_t* R = P + s.off_R(l);
    if (mix32(C, R, nullptr))
      launch_early(k_mix_fwd32, (s.K + MK - 1) / MK, TB, 0, st, shat, reinterpret_cast<const uint4*>(R), w.c, s.K);
    else
      k_mix_fwd<<<warps_grid, TB, 0, st>>>(shat, R, w.c, C, s.K);
    idft3(s, w, w.c, zl, w.v + (l + 1) * CV, false, l + 1 < s.L ? 1 : 2, st);
  }
  pw(w.v + s.L * CV, C, P + s.off_Q(), P + s.off_q(), 3, y, V, 0, st);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int mond_fno_backward(mond_fno_shape sh, const uint16_t* P, const float* x, const float* dy, float* grad,
                      void* workspace, void* stream) {
  Shape s;
  if (!P || !x || !dy || !grad || !workspace || !make_shape(sh, &s)) return -1;
  cudaStream_t st = (cudaStream_t)stream;
  if (!smem_opt_in()) return -3;
  Work w;
  carve(s, (char*)workspace, &w);
  const int C = s.C, M = s.M;
  const int64_t V = s.V, CV = (int64_t)C * V;
  const unsigned gw = (unsigned)std::min<int64_t>(V / 64, 152);
  const unsigned warps_grid = (unsigned)(((int64_t)s.K * 32 + TB - 1) / TB);
  // projection
  launch_early(k_wgrad, gw, TB, 0, st, dy, 3, w.v + s.L * CV, C, V, grad + s.off_Q(), grad + s.off_q(),
               aligned16(dy) && aligned16(w.v + s.L * CV));
  float* dv = w.dv;
  float* dv2 = w.dv2;
  pw(dy, 3, P + s.off_Q(), nullptr, C, dv, V, 1, st);
  for (int l = s.L - 1; l >= 0; l--) {
    const float* vl = w.v + l * CV;
    const float* zl = w.z + l * CV;
    const float* dz = dv;  // the last layer has no activation
    if (l + 1 < s.L) {
      launch_early(k_gelu_bwd, grid_stride(CV / 4), TB, 0, st, reinterpret_cast<const float4*>(zl),
                   reinterpret_cast<const float4*>(dv), reinterpret_cast<float4*>(w.dz), CV / 4);
      dz = w.dz;
    }
    // pointwise part
    launch_early(k_wgrad, gw, TB, 0, st, dz, C, vl, C, V, grad + s.off_W(l), grad + s.off_b(l),
                 aligned16(dz) && aligned16(vl));
    pw(dz, C, P + s.off_W(l), nullptr, C, dv2, V, 1, st);
    // spectral part: G_t = (a/V) DFT(dz), through the mixing adjoint, back with the adjoint transform
    dft3(s, w, dz, w.c, st);
    const float2* shat = w.shat + (int64_t)l * C * s.K;
    const uint16_t* R = P + s.off_R(l);
    float* dR = grad + s.off_R(l);
    if (mix32(C, R, dR))
      launch_early(k_mix_bwd32, (s.K + MK - 1) / MK, TB, 0, st, w.c, shat, reinterpret_cast<const uint4*>(R), w.d,
                   reinterpret_cast<float4*>(dR), s.K, M, 1.f / (float)V);
    else
      k_mix_bwd<<<warps_grid, TB, 0, st>>>(w.c, shat, R, w.d, dR, C, s.K, M, 1.f / (float)V);
    idft3(s, w, w.d, dv2, nullptr, true, 0, st);
    float* t = dv;
    dv = dv2;
    dv2 = t;
  }
  // lift
  launch_early(k_wgrad, gw, TB, 0, st, dv, C, x, 4, V, grad + s.off_P(), grad + s.off_p(),
               aligned16(dv) && aligned16(x));
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int mond_fno_loss(int64_t count, const float* y, const float* t, float* dy, float weight, double* loss_acc,
                  void* stream) {
  if (!y || !t || !dy || !loss_acc || count <= 0) return -1;
  cudaStream_t st = (cudaStream_t)stream;
  double* tn = loss_acc + 1;  // scratch slot after the accumulator
  cudaMemsetAsync(tn, 0, sizeof(double), st);
  sumsq(t, count, tn, st);
  launch_early(k_loss, grid_stride(count), TB, 0, st, y, t, dy, count, tn, weight, loss_acc);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int mond_fno_adam_cast(int64_t count, float* p, float* g, float* m, float* v, float lr, float b1, float b2, float eps,
                       int step, float clip_norm, double* scratch, uint16_t* pb, void* stream) {
  if (!p || !g || !m || !v || count <= 0 || step < 1 || !scratch) return -1;
  cudaStream_t st = (cudaStream_t)stream;
  const AdamArgs a{lr, b1, b2, eps, 1.f - powf(b1, (float)step), 1.f - powf(b2, (float)step), clip_norm, scratch};
  cudaMemsetAsync(scratch, 0, sizeof(double), st);
  const unsigned grid = grid_stride((count + 3) / 4);
  sumsq(g, count, scratch, st);
  const int vec = aligned16(p) && aligned16(g) && aligned16(m) && aligned16(v) &&
                  (reinterpret_cast<uintptr_t>(pb) & 7) == 0;
  launch_early(k_adam, vec ? grid : grid_stride(count), TB, 0, st, count, p, g, m, v, pb, a, vec);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int mond_fno_adam(int64_t count, float* p, float* g, float* m, float* v, float lr, float b1, float b2, float eps,
                  int step, float clip_norm, double* scratch, void* stream) {
  return mond_fno_adam_cast(count, p, g, m, v, lr, b1, b2, eps, step, clip_norm, scratch, nullptr, stream);
}

int mond_fno_coarsen(int N, int n, int ncomp, const float* fine, const float* fine2, float* coarse,
                     const float* scale, void* stream) {
  if (!fine || !coarse || n <= 0 || N % n || ncomp < 1) return -1;
  launch_coarsen(N, n, ncomp, fine, fine2, coarse, scale, (cudaStream_t)stream);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int mond_fno_input(int N, int n, float a0, const float* gN, float* x, float* scale_out, void* stream) {
  if (!gN || !x || !scale_out || n <= 0 || N % n) return -1;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t V = (int64_t)n * n * n;
  // coarse g_N into the x buffer's first 3 planes, its sum of squares into the scale slot's neighbour
  launch_coarsen(N, n, 3, gN, nullptr, x, nullptr, st);
  double* acc = reinterpret_cast<double*>(scale_out + 2);  // scale_out must have room for 2 + 2 floats
  cudaMemsetAsync(acc, 0, sizeof(double), st);
  sumsq(x, 3 * V, acc, st);
  launch_early(k_input, grid_stride(V), TB, 0, st, n, a0, x, acc, x, scale_out);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

size_t mond_fno_output_scratch_bytes(int N, int n) {
  if (n <= 0 || N % n) return 0;
  return sizeof(float) * 3 * ((size_t)n * n * N + (size_t)n * N * N);
}

int mond_fno_output(int N, int n, const float* y, const float* scale, float* H, void* scratch, void* stream) {
  if (!y || !scale || !H || !scratch || n <= 0 || N % n) return -1;
  const int f = N / n;
  if (f > 64) return -1;
  cudaStream_t st = (cudaStream_t)stream;
  if (f % 4 == 0 && n % 4 == 0 && N <= 512 && aligned16(y) && aligned16(H)) {
    launch_early(k_up3, dim3(n, n / UPZ, 3 * (f / 4)), dim3(N / 4, 256 / (N / 4)), smem_up3(n, N), st, n, N,
                 reinterpret_cast<const float4*>(y), reinterpret_cast<float4*>(H), scale);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
  }
  float* t1 = (float*)scratch;              // [3 n n][N]   x upsampled
  float* t2 = t1 + (size_t)3 * n * n * N;   // [3 n][N][N]  x, y upsampled
  const int threads = N < 256 ? ((N + 31) / 32) * 32 : 256;
  k_up_x<<<(unsigned)(3 * n * n), threads, 0, st>>>(n, N, y, t1);
  const size_t wsm = sizeof(float) * 4 * f;
  const int64_t inner2 = (int64_t)N * N, chunk2 = inner2 < 2048 ? inner2 : 2048;
  k_up_axis<<<dim3((unsigned)(3 * n * n), 1), threads, wsm, st>>>(n, N, N, N, t1, t2, nullptr);
  k_up_axis<<<dim3((unsigned)(3 * n), (unsigned)((inner2 + chunk2 - 1) / chunk2)), 256, wsm, st>>>(
      n, N, inner2, chunk2, t2, H, scale);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int mond_fno_mixture_density(int N, double s, int K, const float* centre, const float* mass, const float* radius,
                             const int* kind, float rmax, float* rho, void* stream) {
  if (!centre || !mass || !radius || !kind || !rho || K < 1 || N < 8) return -1;
  k_mixture<<<grid_stride((int64_t)N * N * N), TB, 0, (cudaStream_t)stream>>>(N, (float)s, K, centre, mass, radius,
                                                                             kind, rmax, rho);
  return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // extern "C"
