// particles.cuh -- particle-side kernels: binning by mesh tile, the
// fixed-point deposit of Eq. smooth (Sect. 3.1), the gather of Eq. gi with the
// leapfrog of Eq. motion, and FP64 particle diagnostics.
#pragma once
#include <type_traits>

#include "common.cuh"
#include "fixed_point.cuh"
#include "tma.cuh"

namespace parts {

constexpr int TILE = 8;       // mesh tile side: work items never span two tiles
constexpr int DEP_NT = 256;   // threads per deposit CTA
constexpr int CHUNK = 1024;   // default particles per work item (runtime: the args' chunk)
// Tiles with fewer particles make no work item: their particles are dealt to
// the warps one by one and work on the mesh directly, without a staged copy of
// the tile. Deposit / gather with a limit of 4, 8, 12, 16, 24, 32 particles:
// 0.90 / 0.75, 0.86 / 0.70, 0.83 / 0.73, 0.82 / 0.75, 0.82 / 0.83, 0.79 / 1.02
// ms for 1e6 particles of an isothermal sphere on 256^3 (sigma 1.5), and 0.20 /
// 0.16, 0.18 / 0.14, 0.17 / 0.13, 0.17 / 0.13, 0.16 / 0.14, 0.20 / 0.16 ms for
// 4e5 of a Plummer sphere on 192^3 (sigma 1). At sigma 2, 8, 16 and 24: 1.73 /
// 1.35, 1.69 / 1.30, 1.74 / 1.34 ms for 1e6 on 256^3; only where all tiles hold
// about as many as the limit does it matter (6e4 uniform on 128^3, 15 a
// tile: sigma 2 0.40 / 0.32, 0.49 / 0.41, 0.60 / 0.51 ms, sigma 1 0.090
// / 0.078, 0.076 / 0.067, 0.075 / 0.065).
constexpr int SPARSE = 16;
constexpr int SMS = 152;      // SMs of the GPU
constexpr int QHALF = 32768;  // offset quantisation: q = round(offset * 2^16) + 32768
constexpr int SCAN_B = 8192;  // elements per block of the key scan

// Sort key of a cell: tile-major, then the cell inside its 8^3 tile, so the
// particles of one tile are contiguous and, inside it, grouped by cell.
__device__ __forceinline__ uint32_t cell_key(int c0, int c1, int c2, int ntx) {
  uint32_t t = (uint32_t)(((c2 >> 3) * ntx + (c1 >> 3)) * ntx + (c0 >> 3));
  return t * 512u + (uint32_t)(((c2 & 7) * 8 + (c1 & 7)) * 8 + (c0 & 7));
}

// The deposit's and the gather's work, made by the binning. A work item is a
// run of sorted particles of one tile, {tile, first, past the last, 0}: items
// of `chunk` particles from the front of the array, the tiles' remainders from
// its back, so that the longest start first. The sorted positions of the
// particles of sparse tiles are listed one by one. count: [0] full items,
// [1] remainders, [2] listed particles (zeroed before the binning).
struct Work {
  int4* items;
  int cap;         // entries of items
  uint32_t* list;  // N entries (the keys' memory, free after the sort)
  int* count;
};

struct BinArgs {
  int n, ntx, ntile;
  int64_t ncell;  // n^3 (the key of an invalid particle)
  int64_t N;
  const int32_t* cell;
  const float* off;
  const float* mass;
  uint32_t* key;
  int* count;        // ncell + 1 counters (cleared before)
  int* cstart;       // ncell + 2: first sorted position of each key
  int* bsum;         // per-block sums of the scan
  int* tile_start;   // ntile + 1
  Work work;         // the work list this binning makes
  int chunk;         // particles per work item
  uint32_t* perm;
  uint32_t* status;
};

// Key of each particle, or ncell when it is invalid (cell outside [0, n),
// offset outside [-1/2, 1/2] or not finite, mass not finite).
__global__ void k_bin_count(BinArgs a) {
  kernel_wait();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.N) return;
  int c[3];
  bool ok = true;
  for (int d = 0; d < 3; d++) {
    c[d] = a.cell[3 * i + d];
    float o = a.off[3 * i + d];
    ok &= (c[d] >= 0 && c[d] < a.n && o >= -0.5f && o <= 0.5f);
  }
  ok &= isfinite(a.mass[i]);
  uint32_t k = ok ? cell_key(c[0], c[1], c[2], a.ntx) : (uint32_t)a.ncell;
  if (!ok) set_status(a.status, ST_DOMAIN);
  a.key[i] = k;
  atomicAdd(&a.count[k], 1);
}

__device__ __forceinline__ int block_excl_scan(int v, int* wsum, int* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  if (w == 0) {
    int y = lane < nw ? wsum[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      int t = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += t;
    }
    wsum[lane] = y;
  }
  __syncthreads();
  int r = (w > 0 ? wsum[w - 1] : 0) + x - v;
  if (total) *total = wsum[nw - 1];
  __syncthreads();
  return r;
}

// Scan of the M = ncell + 1 counters in three launches. First the total of
// each block of SCAN_B counters (16-byte loads, a warp reduction, the warps'
// sums in shared memory).
__global__ void __launch_bounds__(1024) k_scan_reduce(const int* cnt, int64_t M, int* bsum) {
  kernel_wait();
  __shared__ int wsum[32];
  const int64_t b0 = (int64_t)blockIdx.x * SCAN_B;
  int s = 0;
  if (b0 + SCAN_B <= M) {
    const int4* c4 = reinterpret_cast<const int4*>(cnt + b0);
    for (int k = threadIdx.x; k < SCAN_B / 4; k += 1024) {
      const int4 v = c4[k];
      s += (v.x + v.y) + (v.z + v.w);
    }
  } else {
    for (int k = threadIdx.x; k < SCAN_B; k += 1024)
      if (b0 + k < M) s += cnt[b0 + k];
  }
  s = __reduce_add_sync(0xffffffffu, s);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    int t = threadIdx.x < (int)(blockDim.x >> 5) ? wsum[threadIdx.x] : 0;
    t = __reduce_add_sync(0xffffffffu, t);
    if (threadIdx.x == 0) bsum[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(1024) k_scan_blocks(int* bsum, int nblk) {
  kernel_wait();
  __shared__ int wsum[32];
  const int per = (nblk + 1023) / 1024;
  const int i0 = threadIdx.x * per, i1 = min(nblk, i0 + per);
  int s = 0;
  for (int i = i0; i < i1; i++) s += bsum[i];
  int base = block_excl_scan(s, wsum, nullptr);
  for (int i = i0; i < i1; i++) {
    int v = bsum[i];
    bsum[i] = base;
    base += v;
  }
}

// cnt and cstart may be the same array (each thread reads its run before
// writing it); both 16-byte aligned.
__global__ void __launch_bounds__(1024) k_scan_apply(const int* cnt, int64_t M, const int* bsum, int* cstart) {
  kernel_wait();
  __shared__ int wsum[32];
  constexpr int PER = SCAN_B / 1024;
  static_assert(PER == 8, "two int4 per thread");
  const int64_t b0 = (int64_t)blockIdx.x * SCAN_B + (int64_t)threadIdx.x * PER;
  int v[PER], s = 0;
  if (b0 + PER <= M) {
    const int4 a = reinterpret_cast<const int4*>(cnt + b0)[0], b = reinterpret_cast<const int4*>(cnt + b0)[1];
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
  } else {
#pragma unroll
    for (int k = 0; k < PER; k++) v[k] = (b0 + k < M) ? cnt[b0 + k] : 0;
  }
#pragma unroll
  for (int k = 0; k < PER; k++) s += v[k];
  int tot;
  int base = block_excl_scan(s, wsum, &tot) + bsum[blockIdx.x];
  int o[PER];
#pragma unroll
  for (int k = 0; k < PER; k++) {
    o[k] = base;
    base += v[k];
  }
  if (b0 + PER <= M) {
    reinterpret_cast<int4*>(cstart + b0)[0] = make_int4(o[0], o[1], o[2], o[3]);
    reinterpret_cast<int4*>(cstart + b0)[1] = make_int4(o[4], o[5], o[6], o[7]);
  } else {
#pragma unroll
    for (int k = 0; k < PER; k++)
      if (b0 + k < M) cstart[b0 + k] = o[k];
  }
  if (b0 <= M - 1 && M - 1 < b0 + PER) cstart[M] = base;  // the thread holding the last key writes the total
}

// Particles -> sorted positions (the order inside a cell is immaterial).
__global__ void k_bin_scatter(BinArgs a) {
  kernel_wait();
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.N) return;
  uint32_t k = a.key[i];
  int old = atomicSub(&a.count[k], 1);
  a.perm[a.cstart[k] + old - 1] = (uint32_t)i;
}

// Tile ranges and the work list, one thread per tile (the tile starts sit 512
// cells apart in the cell scan, so the reads are spread out). A warp reserves
// its entries with one atomic per counter.
__global__ void __launch_bounds__(256) k_tile_work(BinArgs a) {
  kernel_wait();
  const int t = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  int ts = 0, te = 0;
  if (t < a.ntile) {
    ts = a.cstart[(int64_t)t * 512];
    te = a.cstart[(int64_t)(t + 1) * 512];
    a.tile_start[t] = ts;
  }
  if (t == 0) a.tile_start[a.ntile] = a.cstart[a.ncell];
  const int n = te - ts;
  const bool sparse = n < SPARSE;
  const int v[3] = {sparse ? 0 : n / a.chunk, (!sparse && n % a.chunk) ? 1 : 0, sparse ? n : 0};
  int at[3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    int x = v[k];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    int base = 0;
    if (lane == 31 && x) base = atomicAdd(a.work.count + k, x);
    at[k] = __shfl_sync(0xffffffffu, base, 31) + x - v[k];
  }
  for (int k = 0; k < v[0]; k++) a.work.items[at[0] + k] = make_int4(t, ts + k * a.chunk, ts + (k + 1) * a.chunk, 0);
  if (v[1]) a.work.items[a.work.cap - 1 - at[1]] = make_int4(t, te - n % a.chunk, te, 0);
  for (int k = 0; k < v[2]; k++) a.work.list[at[2] + k] = (uint32_t)(ts + k);
}

// The items a CTA works on, taken from a counter by thread 0. The record of the
// next item (copied asynchronously into one of two shared slots) and the index
// of the one after it are fetched while an item is worked on, so that neither
// the counter's nor the list's latency is waited for.
struct ItemQueue {
  const Work& w;
  int* counter;
  int4* slots;  // two, shared
  int next = 0, b = 0;
  __device__ __forceinline__ void fetch() {
    const int nfull = __ldg(w.count), total = nfull + __ldg(w.count + 1);
    if (next < total) tma::async_copy16(slots + b, w.items + (next < nfull ? next : w.cap - 1 - (next - nfull)));
    else slots[b] = make_int4(-1, 0, 0, 0);
    next = atomicAdd(counter, 1);
  }
  __device__ __forceinline__ ItemQueue(const Work& work, int* c, int4* s) : w(work), counter(c), slots(s) {
    if (threadIdx.x == 0) {
      next = atomicAdd(counter, 1);
      fetch();
    }
  }
  // the next item for all threads of the CTA (tile -1: none left); a barrier
  __device__ __forceinline__ int4 take() {
    if (threadIdx.x == 0) tma::async_wait_all();
    __syncthreads();
    const int4 it = slots[b];
    b ^= 1;
    if (threadIdx.x == 0 && it.x >= 0) fetch();
    return it;
  }
};

// ---------------------------------------------------------------------------
// Fixed-point deposit.
// ---------------------------------------------------------------------------
struct DepArgs {
  int n, ntx, ntile, r, nb;
  const int32_t* cell;
  const float* off;
  const float* mass;
  const uint32_t* perm;
  Work work;
  const uint32_t* lut;      // (65537) rows of axis_pitch(r) words (2r+1 used), row q + 32768
  const uint32_t* ball;     // packed (dx+r) | (dy+r) << 8 | (dz+r) << 16
  const int32_t* rows;      // dy | dz << 8 | L << 16 of each row (shifted by r), see Rows
  int nrows;                // rows (dy, dz) of the ball
  uint64_t* dep;
  int kacc;
  uint32_t max_sum;   // particles whose taps' upper product words fit one 32-bit sum
  int* work_counter;  // persistent-grid work queues, items and listed particles (zeroed before launch)
};

// 64-bit add into a shared accumulator held as three 32-bit words of 20-bit
// digits, value = s0 + s1 2^20 + s2 2^40 (mod 2^64). The adds need no return
// value (no carry chain); s0 and s1 take at most 4096 addends of < 2^20 each
// without overflow (a work item holds at most 4096 particles and a particle
// adds to a cell once), and s2 may wrap freely because s2 2^40 is only needed
// modulo 2^64.
__device__ __forceinline__ void sadd2(uint32_t* s, int plane, uint32_t vl, uint32_t vh) {
  atomicAdd(s, vl & 0xFFFFFu);
  atomicAdd(s + plane, __funnelshift_r(vl, vh, 20) & 0xFFFFFu);  // unconditional: a zero add is cheaper than a branch
}
__device__ __forceinline__ void sadd3(uint32_t* s, int plane, uint32_t vl, uint32_t vh) {
  sadd2(s, plane, vl, vh);
  if (vh >> 8) atomicAdd(s + 2 * plane, vh >> 8);
}

// Rows (dy, dz) of the ball per lane, ordered by decreasing x extent L
// (dx in [-L, L]): slot k of a lane holds row lane + 32 k. For a reach R the
// widest ball is |d|^2 < (R + 1)^2; its slot k reaches lmax(k) at most, and so
// does that of every narrower ball of the same reach (the k-th longest row
// only shrinks), so that the taps of a slot are register arrays of a size
// known at compile time.
template <int R>
struct Rows {
  // rows whose extent is at least l
  static constexpr int count(int l) {
    int c = 0;
    for (int z = -R; z <= R; z++)
      for (int y = -R; y <= R; y++)
        if (l * l + y * y + z * z < (R + 1) * (R + 1)) c++;
    return c;
  }
  static constexpr int SLOTS = (count(0) + 31) / 32;
  static constexpr int lmax(int k) {
    int l = 0;
    while (l < R && count(l + 1) > 32 * k) l++;
    return l;
  }
  // the shortest row of slot k of the widest ball (-1: a lane without a row)
  static constexpr int lmin(int k) {
    int l = -1;
    while (l < R && count(l + 1) >= 32 * (k + 1)) l++;
    return l;
  }
  static constexpr int W2 = 2 * R + 1;
};

// Runs f(integral constant k) for k in [K0, K1): register arrays are indexed
// by compile-time values.
template <int K0, int K1, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (K0 < K1) {
    f(std::integral_constant<int, K0>{});
    static_for<K0 + 1, K1>(static_cast<F&&>(f));
  }
}

// Rows of a lane, one word per slot: the y and z word offsets (bytes) of a
// particle's axis tables in the low halves, the row's x extent L above them
// (-1: no such row), so that d <= L is one signed compare of the word.
template <int R>
struct LaneRows {
  int info[Rows<R>::SLOTS];
  __device__ __forceinline__ void init(const int32_t* rows, int nrows, int lane) {
#pragma unroll
    for (int k = 0; k < Rows<R>::SLOTS; k++) {
      const int idx = lane + 32 * k;
      info[k] = idx < nrows ? (__ldg(rows + idx) & 0xFF0000) | (__ldg(rows + idx) & 0xFFFF) * 4 : (int)0xFFFF0000;
    }
  }
  __device__ __forceinline__ int y4(int k) const { return info[k] & 0xFF; }
  __device__ __forceinline__ int z4(int k) const { return (info[k] >> 8) & 0xFF; }
  __device__ __forceinline__ void opaque() {
#pragma unroll
    for (int k = 0; k < Rows<R>::SLOTS; k++) asm volatile("" : "+r"(info[k]));
  }
  __device__ __forceinline__ bool reaches(int k, int d) const { return info[k] >= (d << 16); }
};

// Particles staged per warp and batch, and the words of one particle's axis
// tables (three axes, padded to 16 bytes so that the x weights are read as
// 16-byte broadcasts).
constexpr int BATCH = 16;
constexpr int axis_pitch(int R) { return (2 * R + 1 + 3) & ~3; }

template <int R>
struct DepStage {
  uint32_t w[BATCH][3][axis_pitch(R)];  // mass-folded x words, y and z table words
  int key[BATCH], sh[BATCH], order[BATCH];
  int q[BATCH][3];                      // quantised offsets
  uint32_t msig[BATCH];
};

// Adds (a b + 2^(sh-1)) >> sh to a sum held in two words: the upper word h of
// the rounded product and the rest of it shifted, l >> sh, are summed apart,
// so that the sum is (hi 2^(32-sh) + lo) exactly as long as neither wraps
// (0 < sh < 32; HI: 32 <= sh < 64, where only h is left and goes to lo).
// Five instructions a tap; a 64-bit sum takes seven.
template <bool HI>
__device__ __forceinline__ void tap_add(uint32_t& lo, uint32_t& hi, uint32_t a, uint32_t b, uint32_t rl, uint32_t rh,
                                        uint32_t sh) {
  if constexpr (HI) {
    asm("{\n .reg .u64 p;\n .reg .u32 l, h;\n mul.wide.u32 p, %1, %2;\n mov.b64 {l, h}, p;\n add.cc.u32 l, l, %3;\n"
        " addc.u32 h, h, %4;\n shr.u32 h, h, %5;\n add.u32 %0, %0, h;\n}\n"
        : "+r"(lo)
        : "r"(a), "r"(b), "r"(rl), "r"(rh), "r"(sh));
  } else {
    asm("{\n .reg .u64 p;\n .reg .u32 l, h;\n mul.wide.u32 p, %2, %3;\n mov.b64 {l, h}, p;\n add.cc.u32 l, l, %4;\n"
        " addc.u32 %1, %1, h;\n shr.u32 l, l, %5;\n add.u32 %0, %0, l;\n}\n"
        : "+r"(lo), "+r"(hi)
        : "r"(a), "r"(b), "r"(rl), "r"(sh));
  }
}

// One warp deposits the particles [q0, q1) of a tile, sorted by cell.
//
// What bounds it: integer issue. A lane keeps the sums of its taps in registers
// for as long as the particles stay in one cell and have one shift (masses of
// one binade), at most max_sum of them, and then adds them to the staged tile
// as digits. The earlier kernel split every tap of every particle into digits
// and added those to shared memory: about 35 issue slots a tap against 5 here
// and 12 per tap and cell. With binning's work list (no search for an item's
// tile) 1.42 -> 0.84 ms for 1e6 particles of an isothermal sphere on 256^3
// (sigma 1.5, 895 taps), 5.61 -> 2.66 ms for 1e7 of a mixture of spheres (sigma
// 1, 251 taps), 174 -> 20 us for 10007 on 64^3 (also the smaller work items).
// WIDE: the ball is the widest of its reach, so that the shortest row of each
// slot is known too and taps no row of the slot lacks need no mask.
template <int R, bool WIDE>
__device__ __forceinline__ void deposit_range(const DepArgs& a, int q0, int q1, int ox, int oy, int oz, uint32_t* sd,
                                              LaneRows<R> lr, DepStage<R>* st) {
  using RW = Rows<R>;
  constexpr int W2 = RW::W2, P = axis_pitch(R);
  constexpr int hw = TILE + 2 * R, px = hw + 1, hv = hw * hw * px;
  const int lane = threadIdx.x & 31;
  if (q0 >= q1) return;
  // slot k: sums of the taps dx in [-lmax(k), lmax(k)] about the current cell
  uint32_t lo[RW::SLOTS][W2], hi[RW::SLOTS][W2];
  static_for<0, RW::SLOTS>([&](auto K) {
    constexpr int k = K, Lk = RW::lmax(k);
#pragma unroll
    for (int t = 0; t <= 2 * Lk; t++) lo[k][t] = hi[k][t] = 0u;
  });
  int key = -1;         // cell of the staged tile and shift the sums belong to
  uint32_t summed = 0;  // particles in them
  uint32_t inext = lane < BATCH && q0 + lane < q1 ? __ldg(a.perm + q0 + lane) : 0u;
  int p = BATCH;
  for (int g = q0;; g++, p++) {
    if (p == BATCH && g < q1) {
      // stage the next batch: cells, mass parts and axis tables
      p = 0;
      const int cnt = min(BATCH, q1 - g);
      __syncwarp();
      int k2 = 0;
      if (lane < cnt) {
        const int64_t i = inext;
        uint32_t msig;
        int e2;
        const uint32_t mb = __float_as_uint(__ldg(a.mass + i));
        mass_parts(mb, &msig, &e2);
        const int sh = 40 - a.kacc - e2;
        // key: cell of the staged tile << 8 | sign << 7 | shift (0: out of range)
        k2 = (((a.cell[3 * i + 2] - oz - R) * TILE + a.cell[3 * i + 1] - oy - R) * TILE + a.cell[3 * i] - ox - R) << 8 |
             (int)(mb >> 31) << 7 | (sh > 0 && sh < 64 ? sh : 0);
        st->key[lane] = k2;
        st->sh[lane] = sh;
        st->msig[lane] = msig;
#pragma unroll
        for (int d = 0; d < 3; d++) st->q[lane][d] = __float2int_rn(a.off[3 * i + d] * 65536.0f) + QHALF;
        if (g + BATCH + lane < q1) inext = __ldg(a.perm + g + BATCH + lane);
      }
      // the order of the batch: as sorted, or by key when masses of several
      // binades alternate
      const int k0 = __shfl_sync(0xffffffffu, k2, 0) & 0xFF;
      int rank = lane;
      if (__any_sync(0xffffffffu, lane < cnt && (k2 & 0xFF) != k0)) {
        rank = 0;
        for (int l = 0; l < cnt; l++) {
          const int o = __shfl_sync(0xffffffffu, k2, l);
          rank += o < k2 || (o == k2 && l < lane);
        }
      }
      if (lane < cnt) st->order[rank] = lane;
      __syncwarp();
      // four table words per lane and step
      const int quads = cnt * 3 * (P / 4);
      constexpr int UN = (BATCH * 3 * (P / 4) + 31) / 32;
      uint4 t[UN];
#pragma unroll
      for (int u = 0; u < UN; u++) {
        const int e = lane + 32 * u;
        if (e < quads) {
          const int pa = e / (P / 4);
          t[u] = __ldg(reinterpret_cast<const uint4*>(a.lut) + (&st->q[0][0])[pa] * (P / 4) + e - pa * (P / 4));
        }
      }
#pragma unroll
      for (int u = 0; u < UN; u++) {
        const int e = lane + 32 * u;
        if (e < quads) {
          const int pa = e / (P / 4), pp = pa / 3;
          if (pa == 3 * pp) {
            const uint32_t ms = st->msig[pp];
            t[u] = make_uint4(fold_x(t[u].x, ms), fold_x(t[u].y, ms), fold_x(t[u].z, ms), fold_x(t[u].w, ms));
          }
          reinterpret_cast<uint4*>(&st->w[0][0][0])[e] = t[u];
        }
      }
      __syncwarp();
    }
    // what follows from the rows is recomputed per particle: kept in registers
    // across the loop it would spill the sums
    lr.opaque();
    const int pi = g < q1 ? st->order[p] : 0;
    const int nk = g < q1 ? st->key[pi] : -1;  // the last round only empties the sums
    // (a shift below 7 leaves more than 25 bits in the lower sums)
    if (nk != key || summed >= a.max_sum || ((key & 0xF8) == 0 && summed >> (key & 7))) {
      if (key >= 0) {
        const int c = key >> 8, e = 32 - (key & 31);
        const int at = ((c >> 6) * hw + ((c >> 3) & 7)) * px + (c & 7) + R;
        static_for<0, RW::SLOTS>([&](auto K) {
          constexpr int k = K, Lk = RW::lmax(k);
          uint32_t* row = sd + at + ((lr.z4(k) * hw + lr.y4(k)) * px >> 2);
          // a tap past the end of a row adds 0; lanes without a row leave the slot out
          if ((WIDE && RW::lmin(k) >= 0) || lr.reaches(k, 0)) {
            uint32_t top = 0u;
#pragma unroll
            for (int t = 0; t <= 2 * Lk; t++) {
              const uint64_t v = ((uint64_t)hi[k][t] << e) + lo[k][t];
              lo[k][t] = (uint32_t)v;
              hi[k][t] = (uint32_t)(v >> 32);
              sadd2(row + t - Lk, hv, lo[k][t], hi[k][t]);
              top |= hi[k][t];
            }
            if (top >> 8) {
#pragma unroll
              for (int t = 0; t <= 2 * Lk; t++) atomicAdd(row + t - Lk + 2 * hv, hi[k][t] >> 8);
            }
          }
#pragma unroll
          for (int t = 0; t <= 2 * Lk; t++) lo[k][t] = hi[k][t] = 0u;
        });
      }
      key = nk;
      summed = 0;
      if (nk < 0) break;
    }
    const char* wb = reinterpret_cast<const char*>(&st->w[pi][0][0]);
    if ((uint32_t)((key & 0xFF) - 1) < 63u) {
      summed++;
      const uint32_t sh = key & 31;
      uint32_t mx[P];
#pragma unroll
      for (int j = 0; j < P / 4; j++) {
        const uint4 t = reinterpret_cast<const uint4*>(wb)[j];
        mx[4 * j] = t.x, mx[4 * j + 1] = t.y, mx[4 * j + 2] = t.z, mx[4 * j + 3] = t.w;
      }
      auto taps = [&](auto HI, uint32_t rl, uint32_t rh) {
        static_for<0, RW::SLOTS>([&](auto K) {
          constexpr int k = K, Lk = RW::lmax(k);
          const uint32_t rw = row_yz(*reinterpret_cast<const uint32_t*>(wb + 4 * P + lr.y4(k)),
                                     *reinterpret_cast<const uint32_t*>(wb + 8 * P + lr.z4(k)));
#pragma unroll
          for (int d = 0; d <= Lk; d++) {
            // a tap past the end of its row adds the rounded shift of 0, which is 0
            const uint32_t r = (WIDE && d <= RW::lmin(k)) || lr.reaches(k, d) ? rw : 0u;
            tap_add<HI>(lo[k][Lk - d], hi[k][Lk - d], r, mx[R - d], rl, rh, sh);
            if (d) tap_add<HI>(lo[k][Lk + d], hi[k][Lk + d], r, mx[R + d], rl, rh, sh);
          }
        });
      };
      if (!(key & 32)) taps(std::false_type{}, 1u << (sh - 1), 0u);
      else taps(std::true_type{}, sh ? 0u : 0x80000000u, sh ? 1u << (sh - 1) : 0u);
    } else {
      // negative masses, and shifts outside 1..63 (masses changed since they
      // were scanned): tap by tap
      const int c = key >> 8, sh = st->sh[pi];
      for (int t = lane; t < a.nb; t += 32) {
        const uint32_t q = __ldg(a.ball + t);
        const int jx = q & 0xFF, jy = (q >> 8) & 0xFF, jz = (q >> 16) & 0xFF;
        uint64_t v = round_shift((uint64_t)row_yz(st->w[pi][1][jy], st->w[pi][2][jz]) * st->w[pi][0][jx], sh);
        if (key & 0x80) v = 0ull - v;
        sadd3(sd + (((c >> 6) + jz) * hw + ((c >> 3) & 7) + jy) * px + (c & 7) + jx, hv, (uint32_t)v,
              (uint32_t)(v >> 32));
      }
    }
  }
}

// Runs f(first entry, past the last, first step of taps, steps between) over
// the list of the particles of sparse tiles: two entries at a time (one while
// the grid has a warp for each) taken by the grid's warps from a counter, or,
// up to `wide` entries (a CTA for each on the whole GPU), the warps of a CTA
// sharing its taps (a system of a few particles: the latency of a warp's walk
// over the ball is all its time). The two sum a particle's taps in different
// orders, so the choice is one of the list alone, not of the CTAs launched.
template <typename F>
__device__ __forceinline__ void for_sparse(const int* nsparse, int* counter, int wide, F&& f) {
  const int n = __ldg(nsparse), nw = blockDim.x >> 5;
  if (n <= wide) {
    for (int r = blockIdx.x; r < n; r += gridDim.x) {
      if (r != (int)blockIdx.x) __syncthreads();  // the CTA's sums of the entry before have been read
      f(r, r + 1, threadIdx.x >> 5, nw);
    }
    return;
  }
  const int run = n <= (int)gridDim.x * nw ? 1 : 2;
  while (true) {
    int r = 0;
    if ((threadIdx.x & 31) == 0) r = atomicAdd(counter, run);
    r = __shfl_sync(0xffffffffu, r, 0);
    if (r >= n) break;
    f(r, min(n, r + run), 0, 1);
  }
}

// f(in the ball, dx + R, dy + R, dz + R, mesh index) for the taps of the ball
// about a cell, 32 at a time, lanes along the ball's order (x fastest); lanes
// past the last tap repeat it. Branch-free, so that several steps' loads are
// in flight together.
template <int R, typename F>
__device__ __forceinline__ void for_taps(const uint32_t* __restrict__ ball, int nb, int n, int cx, int cy, int cz,
                                         int first, int step, F&& f) {
  const int lane = threadIdx.x & 31;
#pragma unroll 8
  for (int t0 = 32 * first; t0 < nb; t0 += 32 * step) {
    const int t = t0 + lane;
    const uint32_t b = __ldg(ball + min(t, nb - 1));
    const int jx = b & 0xFF, jy = (b >> 8) & 0xFF, jz = b >> 16;
    int gx = cx + jx - R, gy = cy + jy - R, gz = cz + jz - R;
    gx += gx < 0 ? n : (gx >= n ? -n : 0);
    gy += gy < 0 ? n : (gy >= n ? -n : 0);
    gz += gz < 0 ? n : (gz >= n ? -n : 0);
    f(t < nb, jx, jy, jz, (gz * n + gy) * n + gx);
  }
}

// A listed particle, straight into the mesh: the lanes take the taps of the
// ball in their order, x fastest, so that the adds of a row are contiguous
// (the L2's atomics work by sector).
template <int R>
__device__ __forceinline__ void deposit_sparse(const DepArgs& a, int r0, int r1, int first, int step) {
  constexpr int W2 = 2 * R + 1;
  const int lane = threadIdx.x & 31;
  int c[3] = {0, 0, 0}, q[3] = {QHALF, QHALF, QHALF};
  uint32_t mb = 0u;
  if (r0 + lane < r1) {
    const int64_t i = __ldg(a.perm + a.work.list[r0 + lane]);
#pragma unroll
    for (int d = 0; d < 3; d++) {
      c[d] = a.cell[3 * i + d];
      q[d] = __float2int_rn(a.off[3 * i + d] * 65536.0f) + QHALF;
    }
    mb = __float_as_uint(__ldg(a.mass + i));
  }
  for (int p = 0; p < r1 - r0; p++) {
    const int cx = __shfl_sync(0xffffffffu, c[0], p), cy = __shfl_sync(0xffffffffu, c[1], p),
              cz = __shfl_sync(0xffffffffu, c[2], p);
    const uint32_t m = __shfl_sync(0xffffffffu, mb, p);
    uint32_t msig;
    int e2;
    mass_parts(m, &msig, &e2);
    const int sh = 40 - a.kacc - e2;
    uint32_t wt[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const int qd = __shfl_sync(0xffffffffu, q[d], p);
      wt[d] = lane < W2 ? __ldg(a.lut + qd * axis_pitch(R) + lane) : 0u;
    }
    wt[0] = fold_x(wt[0], msig);
    for_taps<R>(a.ball, a.nb, a.n, cx, cy, cz, first, step, [&](bool in, int jx, int jy, int jz, int g) {
      const uint32_t mx = __shfl_sync(0xffffffffu, wt[0], jx), wy = __shfl_sync(0xffffffffu, wt[1], jy),
                     wz = __shfl_sync(0xffffffffu, wt[2], jz);
      uint64_t v = round_shift((uint64_t)row_yz(wy, wz) * mx, sh);
      if (m >> 31) v = 0ull - v;
      if (in && v) atomicAdd((unsigned long long*)(a.dep + g), (unsigned long long)v);
    });
  }
}

// Persistent deposit: CTAs take work items (chunks of up to `chunk` cell-sorted
// particles of one tile) from a counter and accumulate them, a contiguous
// slice per warp, into a shared copy of the tile plus its reach, which is added
// to the global accumulator once. The particles of tiles with too few for that
// follow, straight into the global accumulator.
constexpr int dep_ctas(int R) { return R <= 2 ? 3 : (R <= 5 ? 2 : 1); }
template <int R, bool WIDE>
__global__ void __launch_bounds__(DEP_NT, dep_ctas(R)) k_deposit(DepArgs a) {
  extern __shared__ __align__(16) uint32_t dsm[];
  __shared__ int4 s_items[2];
  constexpr int hw = TILE + 2 * R;
  constexpr int px = hw + 1;  // odd x pitch of the staged tile: rows of different lanes spread over the banks
  constexpr int hv = hw * hw * px;
  DepStage<R>* stage = reinterpret_cast<DepStage<R>*>(dsm);
  uint32_t* sd = dsm + (DEP_NT / 32) * sizeof(DepStage<R>) / 4;  // the digit planes of the tile accumulator
  LaneRows<R> lr;
  lr.init(a.rows, a.nrows, threadIdx.x & 31);
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  ItemQueue queue(a.work, a.work_counter, s_items);
  while (true) {
    const int4 item = queue.take();
    const int t = item.x, p0 = item.y, p1 = item.z;
    if (t < 0) break;
    const int tx = t % a.ntx, ty = (t / a.ntx) % a.ntx, tz = t / (a.ntx * a.ntx);
    const int ox = tx * TILE - R, oy = ty * TILE - R, oz = tz * TILE - R;
    const int len = (p1 - p0 + nw - 1) / nw;
    const int q0 = min(p1, p0 + warp * len), q1 = min(p1, q0 + len);
    for (int k = threadIdx.x; k < (3 * hv + 3) / 4; k += blockDim.x)
      reinterpret_cast<uint4*>(sd)[k] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    deposit_range<R, WIDE>(a, q0, q1, ox, oy, oz, sd, lr, stage + warp);
    __syncthreads();
    const bool inside = ox >= 0 && oy >= 0 && oz >= 0 && ox + hw <= a.n && oy + hw <= a.n && oz + hw <= a.n;
    for (int e = threadIdx.x; e < hw * hw * hw; e += blockDim.x) {
      const int lx = e % hw, row = e / hw, ly = row % hw, lz = row / hw, k = row * px + lx;
      const unsigned long long v = (unsigned long long)sd[k] + ((unsigned long long)sd[hv + k] << 20) +
                                   ((unsigned long long)sd[2 * hv + k] << 40);
      if (v == 0ull) continue;
      int gx = ox + lx, gy = oy + ly, gz = oz + lz;
      if (!inside) {
        gx += gx < 0 ? a.n : (gx >= a.n ? -a.n : 0);
        gy += gy < 0 ? a.n : (gy >= a.n ? -a.n : 0);
        gz += gz < 0 ? a.n : (gz >= a.n ? -a.n : 0);
      }
      atomicAdd((unsigned long long*)(a.dep + (gz * a.n + gy) * a.n + gx), v);
    }
  }
  for_sparse(a.work.count + 2, a.work_counter + 1, SMS * dep_ctas(R),
             [&](int r0, int r1, int first, int step) { deposit_sparse<R>(a, r0, r1, first, step); });
}
template <int R>
constexpr size_t dep_smem_bytes() {
  constexpr size_t hw = TILE + 2 * R;
  return (DEP_NT / 32) * sizeof(DepStage<R>) + (sizeof(uint32_t) * 3 * hw * hw * (hw + 1) + 15) / 16 * 16;
}

// ---------------------------------------------------------------------------
// Gather (Eq. gi) and leapfrog (Eq. motion).
// ---------------------------------------------------------------------------
struct GatArgs {
  int n, ntx, ntile, r, nb;
  int32_t* cell;
  float* off;
  float* vel;
  const uint32_t* perm;
  const int* tile_start;
  Work work;
  const float* acc;       // 3 real planes
  const uint32_t* ball;
  const int32_t* rows;    // as in DepArgs
  int nrows;              // rows (dy, dz) of the ball
  float* g_out;           // optional [N][3] force output
  float dt;               // kick time step
  float dt_over_s;        // drift: offset += v dt / s
  int do_kick, do_drift;
  float inv2s2;           // 1 / (2 sigma^2)
  float gnorm;            // 1 / (sigma sqrt(2 pi))
  int* work_counter;      // as in DepArgs
  uint32_t* status;
};

// Leapfrog of one particle axis: component ax of particle i, force g, cell c,
// offset o, velocity v.
__device__ __forceinline__ void gather_push1(const GatArgs& a, int64_t i, int ax, float g, int c, float o, float v) {
  if (a.g_out) a.g_out[3 * i + ax] = g;
  if (!isfinite(g)) set_status(a.status, ST_NAN);
  if (a.do_kick) {
    v += g * a.dt;
    a.vel[3 * i + ax] = v;
    if (a.do_drift) {
      o += v * a.dt_over_s;
      const float sh = floorf(o + 0.5f);
      c += (int)sh;
      c += c < 0 ? a.n : (c >= a.n ? -a.n : 0);
      a.off[3 * i + ax] = o - sh;
      a.cell[3 * i + ax] = c;
    }
  }
}

// A load that stays where it is written (ahead of the work that hides it; the
// compiler otherwise moves it down to its use to save a register).
__device__ __forceinline__ int load_now(const int* p) {
  int v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Particles per warp and batch of the gather (3 lanes each), and the words of
// a row of lane sums (padded to spread 16-byte reads over the banks).
constexpr int GBATCH = 10;
constexpr int GSUM = 36;

template <int R>
struct GatStage {
  float w[GBATCH][3][axis_pitch(R)];  // axis weights
  float sum[3 * GBATCH][GSUM];        // per particle and axis: the lanes' partial sums
  int cell[GBATCH][4];
  float off[GBATCH][4];
};

// Slots [K0, K1) of the rows of one cell held in registers at a time: all of
// them up to reach 5 (34 taps x 3 components), fewer per pass beyond.
template <int R>
struct GatPasses {
  static constexpr int N = R <= 5 ? 1 : (R == 6 ? 2 : 3);
  static constexpr int first(int p) { return p >= N ? Rows<R>::SLOTS : 2 * p; }
};

// One warp gathers the particles [q0, q1) of a tile, sorted by cell.
//
// What bounds it: shared-memory reads and FP32 issue. A lane reads the taps of
// its rows about a cell once, into registers, and uses them for every particle
// of the cell (the earlier kernel read each tap from shared memory for every
// pair of particles). Taps outside the ball are held as 0. A lane's sums of a
// particle go to shared memory and are added over the lanes for GBATCH
// particles at a time, 32 values by one lane, instead of a shuffle reduction
// per particle; the lane that adds them kicks and drifts that axis. Added one
// after the other they raised the rms error of a force by 4 to 6%; pairwise, in
// 0.3% more time, it is that of the reduction (1.18, 1.25, 1.12 and 1.22e-7 at
// sigma 0.75, 1, 1.5 and 2). 0.93 ->
// 0.66 ms for 1e6 particles of an isothermal sphere on 256^3 (sigma 1.5), 3.56
// -> 1.99 ms for 1e7 of a mixture of spheres (sigma 1), 77 -> 18 us for 10007
// on 64^3.
template <int R>
__device__ __forceinline__ void gather_range(const GatArgs& a, int q0, int q1, int ox, int oy, int oz,
                                             const float2* sa, const float* sz, LaneRows<R> lr, GatStage<R>* st) {
  using RW = Rows<R>;
  using GP = GatPasses<R>;
  constexpr int W2 = RW::W2, P = axis_pitch(R);
  constexpr int hw = TILE + 2 * R, px = hw + 1;
  const int lane = threadIdx.x & 31;
  const int lp = lane / 3, lax = lane - 3 * lp;  // the particle of a batch and the axis this lane loads and kicks
  // the inputs of the next batch, and the indices of the one after it, are
  // fetched while a batch is gathered (a particle's cell and offset change only
  // when this warp drifts it)
  int64_t in = 0;
  uint32_t inn = 0u;
  int cn = 0;
  float on = 0.f, vn = 0.f;
  auto fetch = [&](int b) {
    in = inn;
    if (lane < 3 * GBATCH && b + lp < q1) {
      cn = load_now(a.cell + 3 * in + lax);
      on = __int_as_float(load_now(reinterpret_cast<const int*>(a.off) + 3 * in + lax));
      if (a.do_kick) vn = __int_as_float(load_now(reinterpret_cast<const int*>(a.vel) + 3 * in + lax));
    }
  };
  auto fetch_index = [&](int b) {
    if (lane < 3 * GBATCH && b + lp < q1) inn = (uint32_t)load_now(reinterpret_cast<const int*>(a.perm) + b + lp);
  };
  fetch_index(q0);
  fetch(q0);
  fetch_index(q0 + GBATCH);
  for (int b = q0; b < q1; b += GBATCH) {
    const int cnt = min(GBATCH, q1 - b);
    const int64_t i = in;
    const int c = cn;
    const float o = on, v = vn;
    __syncwarp();
    if (lp < cnt) {
      st->cell[lp][lax] = c;
      st->off[lp][lax] = o;
    }
    fetch(b + GBATCH);
    fetch_index(b + 2 * GBATCH);
    __syncwarp();
    for (int e = lane; e < cnt * 3 * W2; e += 32) {
      const int pa = e / W2, j = e - pa * W2, p = pa / 3, ax = pa - 3 * p;
      const float u = (float)(j - R) - st->off[p][ax];
      st->w[p][ax][j] = expf(-u * u * a.inv2s2) * a.gnorm;
    }
    __syncwarp();
    for (int p0 = 0; p0 < cnt;) {
      // the particles p0 .. p1 - 1 share a cell
      const int4 m = *reinterpret_cast<const int4*>(st->cell[p0]);
      int p1 = p0 + 1;
      while (p1 < cnt && st->cell[p1][0] == m.x && st->cell[p1][1] == m.y && st->cell[p1][2] == m.z) p1++;
      static_for<0, GP::N>([&](auto PASS) {
        constexpr int K0 = GP::first(PASS), K1 = GP::first(PASS + 1);
        lr.opaque();
        float tx[K1 - K0][W2], ty[K1 - K0][W2], tz[K1 - K0][W2];
        static_for<K0, K1>([&](auto K) {
          constexpr int k = K, Lk = RW::lmax(k);
          const int row = ((m.z + (lr.z4(k) >> 2) - R - oz) * hw + (m.y + (lr.y4(k) >> 2) - R - oy)) * px + m.x - ox;
#pragma unroll
          for (int x = 0; x <= 2 * Lk; x++) {
            const bool in = lr.reaches(k, x < Lk ? Lk - x : x - Lk);
            const float2 q = in ? sa[row + x - Lk] : make_float2(0.f, 0.f);
            tx[k - K0][x] = q.x;
            ty[k - K0][x] = q.y;
            tz[k - K0][x] = in ? sz[row + x - Lk] : 0.f;
          }
        });
        for (int p = p0; p < p1; p++) {
          const char* wb = reinterpret_cast<const char*>(&st->w[p][0][0]);
          float wx[P];
#pragma unroll
          for (int j = 0; j < P / 4; j++) {
            const float4 q = reinterpret_cast<const float4*>(wb)[j];
            wx[4 * j] = q.x, wx[4 * j + 1] = q.y, wx[4 * j + 2] = q.z, wx[4 * j + 3] = q.w;
          }
          float gx = 0.f, gy = 0.f, gz = 0.f;
          static_for<K0, K1>([&](auto K) {
            constexpr int k = K, Lk = RW::lmax(k);
            const float wyz = *reinterpret_cast<const float*>(wb + 4 * P + lr.y4(k)) *
                              *reinterpret_cast<const float*>(wb + 8 * P + lr.z4(k));
            float sx = 0.f, sy = 0.f, sw = 0.f;
#pragma unroll
            for (int x = 0; x <= 2 * Lk; x++) {
              sx = fmaf(wx[R - Lk + x], tx[k - K0][x], sx);
              sy = fmaf(wx[R - Lk + x], ty[k - K0][x], sy);
              sw = fmaf(wx[R - Lk + x], tz[k - K0][x], sw);
            }
            gx = fmaf(wyz, sx, gx);
            gy = fmaf(wyz, sy, gy);
            gz = fmaf(wyz, sw, gz);
          });
          if constexpr (PASS > 0) {
            gx += st->sum[3 * p][lane];
            gy += st->sum[3 * p + 1][lane];
            gz += st->sum[3 * p + 2][lane];
          }
          st->sum[3 * p][lane] = gx;
          st->sum[3 * p + 1][lane] = gy;
          st->sum[3 * p + 2][lane] = gz;
        }
      });
      p0 = p1;
    }
    __syncwarp();
    if (lp < cnt) {
      // added pairwise, lanes 16 apart first: five roundings deep, as a
      // reduction over the warp
      const float4* q = reinterpret_cast<const float4*>(st->sum[lane]);
      float4 g[4];
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const float4 u = q[j], w = q[j + 4];
        g[j] = make_float4(u.x + w.x, u.y + w.y, u.z + w.z, u.w + w.w);
      }
#pragma unroll
      for (int k = 2; k > 0; k >>= 1)
#pragma unroll
        for (int j = 0; j < k; j++)
          g[j] = make_float4(g[j].x + g[j + k].x, g[j].y + g[j + k].y, g[j].z + g[j + k].z, g[j].w + g[j + k].w);
      gather_push1(a, i, lax, (g[0].x + g[0].z) + (g[0].y + g[0].w), c, o, v);
    }
  }
}

// Listed particles, straight from the mesh: the lanes take the taps of the ball
// in their order, x fastest, so that a row is read by neighbouring lanes; a
// staged tile would cost more than these reads.
template <int R>
__device__ __forceinline__ void gather_sparse(const GatArgs& a, int r0, int r1, int first, int step,
                                              float (*part)[4]) {
  const int lane = threadIdx.x & 31;
  const int n3 = a.n * a.n * a.n;
  int c[3] = {0, 0, 0};
  float o[3] = {0.f, 0.f, 0.f};
  uint32_t idx = 0u;
  if (r0 + lane < r1) {
    idx = __ldg(a.perm + a.work.list[r0 + lane]);
#pragma unroll
    for (int d = 0; d < 3; d++) {
      c[d] = a.cell[3 * (int64_t)idx + d];
      o[d] = a.off[3 * (int64_t)idx + d];
    }
  }
  float g[3] = {0.f, 0.f, 0.f};  // lane p: the force on particle r0 + p
  for (int p = 0; p < r1 - r0; p++) {
    const int cx = __shfl_sync(0xffffffffu, c[0], p), cy = __shfl_sync(0xffffffffu, c[1], p),
              cz = __shfl_sync(0xffffffffu, c[2], p);
    float wt[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const float u = (float)(lane - R) - __shfl_sync(0xffffffffu, o[d], p);
      wt[d] = expf(-u * u * a.inv2s2) * a.gnorm;
    }
    float s[3] = {0.f, 0.f, 0.f};
    for_taps<R>(a.ball, a.nb, a.n, cx, cy, cz, first, step, [&](bool in, int jx, int jy, int jz, int q) {
      // a lane past the last tap repeats it with weight 0
      const float w = __shfl_sync(0xffffffffu, wt[0], jx) *
                      (__shfl_sync(0xffffffffu, wt[1], jy) * __shfl_sync(0xffffffffu, wt[2], jz));
#pragma unroll
      for (int d = 0; d < 3; d++) s[d] = fmaf(in ? w : 0.f, __ldg(a.acc + q + (int64_t)d * n3), s[d]);
    });
#pragma unroll
    for (int d = 0; d < 3; d++) {
      for (int k = 16; k > 0; k >>= 1) s[d] += __shfl_xor_sync(0xffffffffu, s[d], k);
      if (lane == p) g[d] = s[d];
    }
  }
  if (step > 1) {
    // one particle, its taps dealt to the warps of the CTA: lane 0 of warp 0 adds their sums
    if (lane == 0)
      for (int d = 0; d < 3; d++) part[first][d] = g[d];
    __syncthreads();
    if (first > 0) return;
    for (int w = 1; w < step; w++)
      for (int d = 0; d < 3; d++) g[d] += part[w][d];
  }
  if (r0 + lane < r1) {
#pragma unroll
    for (int d = 0; d < 3; d++)
      gather_push1(a, idx, d, g[d], c[d], o[d], a.do_kick ? a.vel[3 * (int64_t)idx + d] : 0.f);
  }
}

// Persistent gather: CTAs take work items (chunks of one tile) from a
// counter, stage the acceleration mesh over the tile plus its reach (periodic
// wrap) in shared memory, one row per warp step, and gather from it; the
// particles of sparse tiles follow. R is the reach of the ball.
constexpr int gat_threads(int R) { return R == 5 ? 192 : 256; }
constexpr int gat_ctas(int R) { return R <= 5 ? 2 : 1; }
template <int R>
constexpr size_t gat_smem_bytes() {
  constexpr size_t hw = TILE + 2 * R;
  return sizeof(float) * ((3 * hw * hw * (hw + 1) + 3) / 4 * 4) + (gat_threads(R) / 32) * sizeof(GatStage<R>);
}
template <int R>
__global__ void __launch_bounds__(gat_threads(R), gat_ctas(R)) k_gather_push(GatArgs a) {
  extern __shared__ __align__(16) float gsm[];
  __shared__ int4 s_items[2];
  constexpr int hw = TILE + 2 * R;
  constexpr int px = hw + 1;  // odd x pitch of the staged tile: rows of different lanes spread over the banks
  // the staged cells: x and y components together, the z component apart (12
  // bytes a cell, so that two CTAs fit where one would with 16)
  float2* sa = reinterpret_cast<float2*>(gsm);
  float* sz = reinterpret_cast<float*>(sa + hw * hw * px);
  GatStage<R>* stage = reinterpret_cast<GatStage<R>*>(gsm + (3 * hw * hw * px + 3) / 4 * 4);
  const int lane = threadIdx.x & 31;
  LaneRows<R> lr;
  lr.init(a.rows, a.nrows, lane);
  const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int n3 = a.n * a.n * a.n;
  ItemQueue queue(a.work, a.work_counter, s_items);
  while (true) {
    const int4 item = queue.take();
    const int t = item.x, p0 = item.y, p1 = item.z;
    if (t < 0) break;
    const int tx = t % a.ntx, ty = (t / a.ntx) % a.ntx, tz = t / (a.ntx * a.ntx);
    const int ox = tx * TILE - R, oy = ty * TILE - R, oz = tz * TILE - R;
    const bool inside = ox >= 0 && oy >= 0 && oz >= 0 && ox + hw <= a.n && oy + hw <= a.n && oz + hw <= a.n;
    for (int e = threadIdx.x; e < hw * hw * hw; e += blockDim.x) {
      const int lx = e % hw, row = e / hw, ly = row % hw, lz = row / hw, k = row * px + lx;
      int gx = ox + lx, gy = oy + ly, gz = oz + lz;
      if (!inside) {
        gx += gx < 0 ? a.n : (gx >= a.n ? -a.n : 0);
        gy += gy < 0 ? a.n : (gy >= a.n ? -a.n : 0);
        gz += gz < 0 ? a.n : (gz >= a.n ? -a.n : 0);
      }
      // asynchronous, so that the whole tile is in flight together
      const float* src = a.acc + (gz * a.n + gy) * a.n + gx;
      tma::async_copy4(&sa[k].x, src);
      tma::async_copy4(&sa[k].y, src + n3);
      tma::async_copy4(sz + k, src + 2 * (int64_t)n3);
    }
    tma::async_wait_all();
    __syncthreads();
    const int len = (p1 - p0 + nw - 1) / nw;
    const int q0 = min(p1, p0 + warp * len), q1 = min(p1, q0 + len);
    gather_range<R>(a, q0, q1, ox, oy, oz, sa, sz, lr, stage + warp);
  }
  __shared__ float part[gat_threads(R) / 32][4];
  for_sparse(a.work.count + 2, a.work_counter + 1, SMS * gat_ctas(R), [&](int r0, int r1, int first, int step) {
    gather_sparse<R>(a, r0, r1, first, step, part);
  });
}

// ---------------------------------------------------------------------------
// Mesh-interpolating gather. The acceleration mesh then holds the
// node-smoothed field (the force Eq. gi gives a particle on each pixel
// centre); the force at a particle is the linear (ORDER 1) or Keys cubic
// (ORDER 3, a = -1/2) interpolation of that field at the particle's position,
// followed by the kick and drift of k_gather_push. One thread per particle, in
// binned order, so that neighbouring threads read neighbouring nodes.
// ---------------------------------------------------------------------------
// Weights of the nodes -1, 0, 1, 2 for a point at fraction t in [0, 1) past
// node 0: Keys' kernel at distances 1 + t, t, 1 - t, 2 - t.
__device__ __forceinline__ void keys_weights(float t, float* w) {
  const float u = 1.0f - t;
  w[1] = (1.5f * t - 2.5f) * t * t + 1.0f;
  w[2] = (1.5f * u - 2.5f) * u * u + 1.0f;
  const float p = 1.0f + t, q = 2.0f - t;
  w[0] = ((-0.5f * p + 2.5f) * p - 4.0f) * p + 2.0f;
  w[3] = ((-0.5f * q + 2.5f) * q - 4.0f) * q + 2.0f;
}

template <int ORDER>
__global__ void __launch_bounds__(256) k_interp_push(GatArgs a) {
  constexpr int NW = ORDER == 3 ? 4 : 2;
  constexpr int LO = ORDER == 3 ? -1 : 0;
  const int nbinned = __ldg(a.tile_start + a.ntile);
  const int n = a.n;
  const int64_t n3 = (int64_t)n * n * n;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nbinned; q += gridDim.x * blockDim.x) {
    const uint32_t i = __ldg(a.perm + q);
    int c[3], b[3];
    float w[3][NW];
#pragma unroll
    for (int ax = 0; ax < 3; ax++) {
      c[ax] = a.cell[3 * i + ax];
      const float o = a.off[3 * i + ax];
      b[ax] = c[ax] + (o < 0.f ? -1 : 0) + LO;
      const float t = o < 0.f ? o + 1.0f : o;
      if constexpr (ORDER == 3) {
        keys_weights(t, w[ax]);
      } else {
        w[ax][0] = 1.0f - t;
        w[ax][1] = t;
      }
    }
    float g0 = 0.f, g1 = 0.f, g2 = 0.f;
#pragma unroll
    for (int dz = 0; dz < NW; dz++) {
      int z = b[2] + dz;
      z += z < 0 ? n : (z >= n ? -n : 0);
#pragma unroll
      for (int dy = 0; dy < NW; dy++) {
        int y = b[1] + dy;
        y += y < 0 ? n : (y >= n ? -n : 0);
        const float wyz = w[1][dy] * w[2][dz];
        const int64_t row = ((int64_t)z * n + y) * n;
#pragma unroll
        for (int dx = 0; dx < NW; dx++) {
          int x = b[0] + dx;
          x += x < 0 ? n : (x >= n ? -n : 0);
          const float wt = w[0][dx] * wyz;
          g0 = fmaf(wt, __ldg(a.acc + row + x), g0);
          g1 = fmaf(wt, __ldg(a.acc + n3 + row + x), g1);
          g2 = fmaf(wt, __ldg(a.acc + 2 * n3 + row + x), g2);
        }
      }
    }
    const float g[3] = {g0, g1, g2};
#pragma unroll
    for (int ax = 0; ax < 3; ax++) {
      if (a.g_out) a.g_out[3 * i + ax] = g[ax];
      if (!isfinite(g[ax])) set_status(a.status, ST_NAN);
      if (a.do_kick) {
        const float v = a.vel[3 * i + ax] + g[ax] * a.dt;
        a.vel[3 * i + ax] = v;
        if (a.do_drift) {
          const float o = a.off[3 * i + ax] + v * a.dt_over_s;
          const float sh = floorf(o + 0.5f);
          int cc = c[ax] + (int)sh;
          cc += cc < 0 ? n : (cc >= n ? -n : 0);
          a.off[3 * i + ax] = o - sh;
          a.cell[3 * i + ax] = cc;
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// FP64 particle diagnostics: slots [0] mass, [1..3] momentum, [4..6] sum m x,
// [7..9] angular momentum about the origin, [10] kinetic energy.
// ---------------------------------------------------------------------------
__global__ void k_particle_diag(int n, double s, int64_t N, const int32_t* cell, const float* off, const float* vel,
                                const float* mass, double* out) {
  double acc[11];
  for (int k = 0; k < 11; k++) acc[k] = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
    double m = mass[i], x[3], v[3];
    for (int d = 0; d < 3; d++) {
      x[d] = ((double)cell[3 * i + d] - n / 2 + (double)off[3 * i + d]) * s;
      v[d] = vel[3 * i + d];
    }
    acc[0] += m;
    for (int d = 0; d < 3; d++) {
      acc[1 + d] += m * v[d];
      acc[4 + d] += m * x[d];
      acc[10] += 0.5 * m * v[d] * v[d];
    }
    acc[7] += m * (x[1] * v[2] - x[2] * v[1]);
    acc[8] += m * (x[2] * v[0] - x[0] * v[2]);
    acc[9] += m * (x[0] * v[1] - x[1] * v[0]);
  }
  for (int k = 0; k < 11; k++) {
    double v = acc[k];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(out + k, v);
  }
}

// Largest biased exponent of |mass| (for the fixed-point scale).
__global__ void k_mass_exponent(int64_t N, const float* mass, int* emax) {
  int e = 1;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
    int b = (__float_as_uint(mass[i]) >> 23) & 0xFF;
    e = max(e, b);
  }
  for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
  if ((threadIdx.x & 31) == 0) atomicMax(emax, e);
}

// Sum over a real plane (FP64), optionally of the product with a second plane.
__global__ void k_plane_sum(int64_t n3, const float* a, const float* b, double* out) {
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += (int64_t)gridDim.x * blockDim.x)
    acc += b ? (double)a[i] * (double)b[i] : (double)a[i];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

}  // namespace parts
