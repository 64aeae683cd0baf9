// linear.cu -- factorised (kernelised) linear attention with phi = elu + 1:
//
//     S = sum_n phi(k_n) v_n^T (d x d),  z = sum_n phi(k_n),
//     out_i = phi(q_i)^T S / (phi(q_i)^T z).
//
// Not an operator of the paper (whose global attention is the tiled GPA): the
// textbook linear-complexity global attention with a fixed-size per-head
// summary and normaliser.  The feature map is the one of Katharopoulos et al.
// (2020).  BF16 inputs, d = 64.
//
// Three kernels, all HBM-bound:
//   la_summary_kernel  split-N summary: each CTA streams a chunk of 128-token
//                      K and V tiles (TMA, 128-byte swizzle) through a ring of
//                      shared-memory stages; eight warps (two per row, 32
//                      columns each) apply phi to the K tile
//                      (rows past N zeroed) and write it as BF16 high parts in
//                      place and low parts (phi - hi) in the stage's third
//                      tile, and accumulate z in FP32 from the unrounded phi;
//                      one thread issues S += phi_hi(K)^T V + phi_lo(K)^T V on
//                      tcgen05 (M = N = 64, both operands MN-major, K = 128
//                      tokens) with the accumulator in TMEM; the CTA writes its
//                      FP32 partial S and z.  (With phi(K) rounded to BF16, S
//                      and z would carry independent 2^-9 per-term errors that
//                      the centred sum of the query gradient amplifies to
//                      ~5e-3 RMS.)
//   la_combine_kernel  per (b, h), the chunk partials summed in fixed order
//                      with Kahan compensation; S^T split into BF16 high and
//                      low parts (S = hi + lo to ~2^-17) for the query pass.
//   la_query_kernel    per 128-token query tile: phi(Q) in place, the
//                      denominator phi(q) . z per row in FP32, O = phi(Q) S on
//                      tcgen05 (two MMAs: hi and lo parts of S), out = O / den.
#include <math.h>

#include "internal.cuh"
#include "sm103_common.cuh"
#include "sm103_ptx.cuh"

GATTN_DEFINE_STATUS(linear)

namespace gattn {
namespace {
using namespace sm103;

constexpr int kD = 64;
constexpr int kTile = 128;                 // tokens per tile
constexpr int kTileBytes = kTile * kD * 2;  // 16 KB, one TMA box
constexpr int kStagesS = 2;                 // summary ring: K (phi hi) + V + phi lo per stage
constexpr int kSumStage = 3 * kTileBytes;
constexpr int kThreadsL = 320;              // producer, issuer, 8 math warps (two per TMEM lane quadrant)
constexpr int kQStages = 2;

__device__ void set_status_l(uint32_t c) { set_status(c); }
#define LWAIT(bar, par) mbar_wait<set_status_l>((bar), (par), abort_flag)
#define WARP_LWAIT(bar, par) warp_ok(LWAIT(bar, par))

__device__ __forceinline__ float phi_f(float x) { return x > 0.f ? x + 1.f : ex2(x * 1.4426950408889634f); }

// phi of the eight BF16 values of one 16-byte chunk, in place; the rounded
// values are also returned as floats.
__device__ __forceinline__ uint4 phi_chunk(uint4 u, bool valid, float (&f)[8]) {
  uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float a = valid ? phi_f(__uint_as_float(w[i] << 16)) : 0.f;
    const float b = valid ? phi_f(__uint_as_float(w[i] & 0xffff0000u)) : 0.f;
    w[i] = pack_bf16(a, b);
    f[2 * i] = __uint_as_float(w[i] << 16);
    f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// byte offset of 16-byte chunk c of row r in a 128-byte-swizzled tile
__device__ __forceinline__ uint32_t swz(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }

// phi of eight BF16 values (unrounded, FP32)
__device__ __forceinline__ void phi8(uint4 u, bool valid, float (&f)[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = valid ? phi_f(__uint_as_float(w[i] << 16)) : 0.f;
    f[2 * i + 1] = valid ? phi_f(__uint_as_float(w[i] & 0xffff0000u)) : 0.f;
  }
}
// BF16 high parts of eight floats and the BF16 low parts (x - hi)
__device__ __forceinline__ void split8(const float (&f)[8], uint4& hi, uint4& lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    h[i] = pack_bf16(f[2 * i], f[2 * i + 1]);
    l[i] = pack_bf16(f[2 * i] - __uint_as_float(h[i] << 16), f[2 * i + 1] - __uint_as_float(h[i] & 0xffff0000u));
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}
// Sums of the 64 columns of a ROWS x 64 matrix in shared memory by THREADS math
// threads (named barrier 1), in a fixed order: thread t adds every
// (THREADS / 64)-th row of column t % 64, then threads 0..63 add those.  The
// result is in threads 0..63.  Rows 0.. of the matrix are overwritten.
template <int THREADS, int ROWS>
__device__ __forceinline__ float column_sum(float* m, int t) {
  constexpr int P = THREADS / 64;
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");  // the rows are written
  float s = 0.f;
#pragma unroll 8
  for (int i = t / 64; i < ROWS; i += P) s += m[i * 64 + (t & 63)];
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");  // the rows are read
  m[t] = s;
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
  if (t >= 64) return 0.f;
  s = 0.f;
#pragma unroll
  for (int p = 0; p < P; ++p) s += m[p * 64 + t];
  return s;
}

// ---- sums over a CTA's tiles.  The tensor core's FP32 accumulator is neither
// compensated nor rounded to nearest, so its error grows with the number of
// products it takes.  It is folded into a compensated sum after every `sum_tiles`
// tiles (LinearPlan), two accumulators in turn so that the products go on
// meanwhile; sum and compensation live in tensor memory, where the M = 64
// accumulator lies: rows 16 q .. 16 q + 15 in lanes 0..15 of lane quadrant q.
// Each of the eight warps that fold takes the 32 columns at its address.
// (16 heads of 262144 tokens in 108 tiles a CTA: S and dS lay 3.0e-5 and 4.6e-5
// from FP64 in relative RMS with one accumulator for all of them, 7.5e-6 and
// 1.2e-5 with a CTA and a partial for every 27, 4.4e-6 and 7.2e-6 with sums of 14;
// 64 heads: 4.1e-5 and 1.3e-4, 3.0e-5 and 4.7e-5, 4.7e-6 and 8.1e-6.  The folds
// cost the forward nothing and the backward 2 %: 770 -> 789 us at 16 heads; a CTA
// for every 27 tiles took 422 us forward and 825 backward, against 398 and 789.)
__device__ __forceinline__ void kahan8(uint32_t (&s)[8], uint32_t (&c)[8], const uint32_t (&x)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float sum = __uint_as_float(s[i]);
    const float y = __uint_as_float(x[i]) - __uint_as_float(c[i]);
    const float t = sum + y;
    c[i] = __float_as_uint((t - sum) - y);
    s[i] = __float_as_uint(t);
  }
}
// accumulator `acc` (its products are complete) into the sum; the first one sets it
__device__ __forceinline__ void fold_sum(uint32_t acc, uint32_t sum, uint32_t comp, bool first) {
#pragma unroll 1  // (registers)
  for (int h = 0; h < 32; h += 8) {
    uint32_t x[8], s[8], c[8];
    tmem_ld8(acc + h, x);
    if (first) {
      tmem_wait_ld(x);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        s[i] = x[i];
        c[i] = 0;
      }
    } else {
      tmem_ld8(sum + h, s);
      tmem_ld8(comp + h, c);
      tmem_wait_ld(x);
      tmem_wait_ld(s);
      tmem_wait_ld(c);
      kahan8(s, c, x);
    }
    tmem_st8(sum + h, s);
    tmem_st8(comp + h, c);
  }
  tmem_wait_st();
}
// the last accumulator and, if there were others, the sum of those: this lane's 32 values
__device__ __forceinline__ void last_sum(uint32_t acc, uint32_t sum, uint32_t comp, bool only, uint32_t (&r)[32]) {
#pragma unroll
  for (int h = 0; h < 32; h += 8) {
    uint32_t x[8], s[8], c[8];
    tmem_ld8(acc + h, x);
    tmem_wait_ld(x);
    if (!only) {
      tmem_ld8(sum + h, s);
      tmem_ld8(comp + h, c);
      tmem_wait_ld(s);
      tmem_wait_ld(c);
      kahan8(s, c, x);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) r[h + i] = only ? x[i] : s[i];
  }
}

struct SumArgs {
  int N, BH, ntiles, chunk_tiles, sum_tiles;
  float* ws_S;  // [chunks, BH, 64, 64]
  float* ws_z;  // [chunks, BH, 64]
};

__global__ void __launch_bounds__(kThreadsL, 2) la_summary_kernel(const __grid_constant__ CUtensorMap tk,
                                                               const __grid_constant__ CUtensorMap tv,
                                                               const SumArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStagesS * kSumStage);
  uint64_t* kready = full + kStagesS;
  uint64_t* empty = kready + kStagesS;
  uint64_t* sfull = empty + kStagesS;  // [2]: an accumulator's last product is complete
  uint64_t* sfree = sfull + 2;         // [2]: it has been folded
  uint64_t* done = sfree + 2;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = blockIdx.x, bh = blockIdx.y;
  const int t0 = chunk * a.chunk_tiles, t1 = min(a.ntiles, t0 + a.chunk_tiles);
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStagesS; ++i) {
      mbar_init(full + i, 1);
      mbar_init(kready + i, 8);
      mbar_init(empty + i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(sfull + i, 1);
      mbar_init(sfree + i, 8);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tk);
    prefetch_tmap(&tv);
  }
  if (warp == 1) {
    tmem_alloc(tslot, 256);  // S accumulators at columns 0 and 64, their sum at 128, its compensation at 192
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {  // ------------------------------------------------ TMA producer
      uint32_t armed = 0, par = 0;
      bool ok = true;
      for (int t = t0, G = 0; t < t1; ++t, ++G) {
        const int st = G % kStagesS, n = G / kStagesS;
        if (!(ok = LWAIT(empty + st, (n & 1) ^ 1))) break;
        mbar_arrive_expect_tx(full + st, 2 * kTileBytes);
        armed |= 1u << st;
        par = (par & ~(1u << st)) | ((n & 1) << st);
        uint8_t* dst = smem + st * kSumStage;
        tma_load_5d(dst, &tk, full + st, 0, t * kTile, 0, 0, bh);
        tma_load_5d(dst + kTileBytes, &tv, full + st, 0, t * kTile, 0, 0, bh);
      }
      if (!ok)
        for (int s = 0; s < kStagesS; ++s)
          if (armed & (1u << s)) mbar_wait<set_status_l>(full + s, (par >> s) & 1, abort_flag, false);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ------------------------------------------------ MMA issuer
      // S[64 x 64] += phi(K)^T V: A = phi(K) tile MN-major (M = d contiguous),
      // B = V tile MN-major (N = d contiguous); a K = 16 step is 16 token rows.
      constexpr uint32_t idS = idesc_bf16(64, 64, 1) | (1u << 15);  // A MN-major
      bool ok = true;
      int m = 0, ch = 0;  // tile within its sum, sum
      for (int t = t0, G = 0; t < t1; ++t, ++G) {
        const int st = G % kStagesS, n = G / kStagesS, b = ch & 1;
        if (!(ok = LWAIT(kready + st, n & 1))) break;
        if (m == 0 && ch >= 2 && !(ok = LWAIT(sfree + b, ((ch >> 1) - 1) & 1))) break;
        tc_fence_after();
        const uint32_t tS = tmem + 64 * b;
        const uint32_t base = smem_u32(smem + st * kSumStage);
        const uint64_t dA = sw128_desc(base, 16384, 1024), dB = sw128_desc(base + kTileBytes, 16384, 1024);
        const uint64_t dAl = sw128_desc(base + 2 * kTileBytes, 16384, 1024);
#pragma unroll
        for (int ks = 0; ks < kTile / 16; ++ks)
          umma_bf16(tS, dmove(dA, ks * 2048), dmove(dB, ks * 2048), idS, (m > 0 || ks > 0) ? 1u : 0u);
#pragma unroll
        for (int ks = 0; ks < kTile / 16; ++ks) umma_bf16(tS, dmove(dAl, ks * 2048), dmove(dB, ks * 2048), idS, 1u);
        umma_commit(empty + st);
        if (++m == a.sum_tiles) {
          umma_commit(sfull + b);
          m = 0;
          ++ch;
        }
      }
      umma_commit(done);
      if (!ok) *abort_flag = 1;
    }
  } else {
    // ------------------------------------------------------------------ phi warps + epilogue
    // two warps per TMEM lane quadrant: this thread's row (token), columns
    // [32 h, 32 h + 32) (chunks 4 h .. 4 h + 3)
    const int quad = warp & 3;
    const int h = (warp - 2) >> 2;
    const int r = quad * 32 + lane;
    float zacc[kD / 2];
#pragma unroll
    for (int i = 0; i < kD / 2; ++i) zacc[i] = 0.f;
    const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16) + 32 * h;
    bool ok = true;
    int m = 0, ch = 0;  // tiles of the current sum, sums folded
    for (int t = t0, G = 0; t < t1; ++t, ++G) {
      const int st = G % kStagesS, n = G / kStagesS;
      if (!(ok = WARP_LWAIT(full + st, n & 1))) break;
      uint8_t* kt = smem + st * kSumStage;
      const bool valid = t * kTile + r < a.N;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint4* p = reinterpret_cast<uint4*>(kt + swz(r, 4 * h + c));
        float f[8];
        phi8(*p, valid, f);
        uint4 hi, lo;
        split8(f, hi, lo);
        *p = hi;
        *reinterpret_cast<uint4*>(kt + 2 * kTileBytes + swz(r, 4 * h + c)) = lo;
#pragma unroll
        for (int e = 0; e < 8; ++e) zacc[c * 8 + e] += f[e];
      }
      fence_proxy_async_smem();  // the tensor core reads what these threads wrote
      __syncwarp();
      if (lane == 0) mbar_arrive(kready + st);
      // the sum that ended with the previous tile, while this tile's products run
      if (m == a.sum_tiles) {
        if (!(ok = WARP_LWAIT(sfull + (ch & 1), (ch >> 1) & 1))) break;
        tc_fence_after();
        fold_sum(tq + 64 * (ch & 1), tq + 128, tq + 192, ch == 0);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(sfree + (ch & 1));
        ++ch;
        m = 0;
      }
      ++m;
    }
    // epilogue: S partial from TMEM (M = 64: rows 16q .. 16q+15 in lanes 0..15
    // of lane quadrant q; this warp's 32 of the 64 columns), z partial reduced
    // over the 128 rows in fixed order
    const bool got = ok && WARP_LWAIT(done, 0);
    tc_fence_after();
    uint32_t s0[32];
    last_sum(tq + 64 * (ch & 1), tq + 128, tq + 192, ch == 0, s0);
    const size_t part = (size_t)chunk * a.BH + bh;
    if (got && lane < 16) {
      float* dst = a.ws_S + (part * kD + quad * 16 + lane) * kD + 32 * h;
#pragma unroll
      for (int j = 0; j < 32; j += 4)
        *reinterpret_cast<float4*>(dst + j) = make_float4(__uint_as_float(s0[j]), __uint_as_float(s0[j + 1]),
                                                          __uint_as_float(s0[j + 2]), __uint_as_float(s0[j + 3]));
    }
    // all stages are idle once `done` completed: reuse them for the z rows
    float* zbuf = reinterpret_cast<float*>(smem);
    if (got) {
#pragma unroll
      for (int i = 0; i < kD / 2; ++i) zbuf[r * kD + 32 * h + i] = zacc[i];
    }
    const float zs = column_sum<256, kTile>(zbuf, threadIdx.x - 64);
    if (got && threadIdx.x - 64 < kD) a.ws_z[part * kD + threadIdx.x - 64] = zs;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
}

// Kahan-compensated sum of n values a `stride` apart in ascending order, the
// loads sixteen at a time: few heads make many chunks, and with one load in
// flight the combine of one head took longer than a tenth of the call.
__device__ __forceinline__ void kahan_chunks(const float* __restrict__ src, size_t stride, int n, float& sum,
                                             float& comp) {
  for (int c0 = 0; c0 < n; c0 += 16) {
    float x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = c0 + i < n ? __ldg(src + (size_t)(c0 + i) * stride) : 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (c0 + i >= n) break;
      const float y = x[i] - comp;
      const float t = sum + y;
      comp = (t - sum) - y;
      sum = t;
    }
  }
}

struct CombArgs {
  int BH, chunks;
  const float* ws_S;
  const float* ws_z;
  __nv_bfloat16* sth;  // [BH, 64 (v), 64 (k)] high part of S^T
  __nv_bfloat16* stl;  // low part
  float* zt;           // [BH, 64]
};

// grid (BH, ceil((64 * 64 + 64) / 256)): one summary entry per thread
__global__ void __launch_bounds__(256) la_combine_kernel(const CombArgs a) {
  const int bh = blockIdx.x;
  for (int e = blockIdx.y * 256 + threadIdx.x; e < kD * kD + kD; e += 256 * gridDim.y) {
    const bool is_z = e >= kD * kD;
    float sum = 0.f, comp = 0.f;  // Kahan
    const float* src = is_z ? a.ws_z + (size_t)bh * kD + (e - kD * kD) : a.ws_S + (size_t)bh * kD * kD + e;
    kahan_chunks(src, (size_t)a.BH * (is_z ? kD : kD * kD), a.chunks, sum, comp);
    if (is_z) {
      a.zt[(size_t)bh * kD + (e - kD * kD)] = sum;
    } else {
      const int k = e / kD, v = e % kD;  // S[k][v] -> S^T[v][k]
      const __nv_bfloat16 hi = __float2bfloat16_rn(sum);
      const __nv_bfloat16 lo = __float2bfloat16_rn(sum - __bfloat162float(hi));
      a.sth[((size_t)bh * kD + v) * kD + k] = hi;
      a.stl[((size_t)bh * kD + v) * kD + k] = lo;
    }
  }
}

struct QArgs {
  int N, BH, ntiles, tiles_per_cta;
  const __nv_bfloat16* sth;
  const __nv_bfloat16* stl;
  const float* zt;
};

constexpr int kThreadsQ = 224;  // producer, issuer, 4 math warps, storer

__global__ void __launch_bounds__(kThreadsQ, 3) la_query_kernel(const __grid_constant__ CUtensorMap tq,
                                                             const __grid_constant__ CUtensorMap to, const QArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sHi = smem;                       // S^T high part, 64 rows x 128 B, swizzled
  uint8_t* sLo = smem + 8192;                // low part
  uint8_t* qst = smem + 16384;               // Q stages
  uint8_t* ost = qst + kQStages * kTileBytes;  // output staging tile (swizzled, TMA store)
  float* zs = reinterpret_cast<float*>(ost + kTileBytes);
  uint64_t* qfull = reinterpret_cast<uint64_t*>(zs + kD);
  uint64_t* aready = qfull + kQStages;
  uint64_t* qempty = aready + kQStages;
  uint64_t* ofull = qempty + kQStages;  // [2]: O double-buffered in TMEM
  uint64_t* ofree = ofull + 2;          // [2]
  uint64_t* sready = ofree + 2;
  uint64_t* staged = sready + 1;
  uint64_t* sfree = staged + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sfree + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.y;
  const int t0 = blockIdx.x * a.tiles_per_cta, t1 = min(a.ntiles, t0 + a.tiles_per_cta);
  if (threadIdx.x == 0) {
    for (int i = 0; i < kQStages; ++i) {
      mbar_init(qfull + i, 1);
      mbar_init(aready + i, 4);
      mbar_init(qempty + i, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(ofull + b, 1);
      mbar_init(ofree + b, 4);
    }
    mbar_init(sready, 4);
    mbar_init(staged, 4);
    mbar_init(sfree, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tq);
    prefetch_tmap(&to);
  }
  if (warp == 1) {
    tmem_alloc(tslot, 128);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {  // ------------------------------------------------ TMA producer
      uint32_t armed = 0, par = 0;
      bool ok = true;
      for (int t = t0, G = 0; t < t1; ++t, ++G) {
        const int st = G % kQStages, n = G / kQStages;
        if (!(ok = LWAIT(qempty + st, (n & 1) ^ 1))) break;
        mbar_arrive_expect_tx(qfull + st, kTileBytes);
        armed |= 1u << st;
        par = (par & ~(1u << st)) | ((n & 1) << st);
        tma_load_5d(qst + st * kTileBytes, &tq, qfull + st, 0, t * kTile, 0, 0, bh);
      }
      if (!ok)
        for (int s = 0; s < kQStages; ++s)
          if (armed & (1u << s)) mbar_wait<set_status_l>(qfull + s, (par >> s) & 1, abort_flag, false);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ------------------------------------------------ MMA issuer
      // O[128 x 64] = phi(Q) S: A = phi(Q) tile K-major, B = S^T rows (K-major),
      // the high and the low BF16 parts of S accumulated in turn.
      constexpr uint32_t idO = idesc_bf16(128, 64, 0);
      const uint64_t dHi = sw128_desc(smem_u32(sHi), 16, 1024), dLo = sw128_desc(smem_u32(sLo), 16, 1024);
      bool ok = LWAIT(sready, 0);
      for (int t = t0, G = 0; t < t1 && ok; ++t, ++G) {
        const int st = G % kQStages, n = G / kQStages;
        const int b = G & 1;
        if (!(ok = LWAIT(aready + st, n & 1))) break;
        if (G >= 2 && !(ok = LWAIT(ofree + b, ((G >> 1) - 1) & 1))) break;
        tc_fence_after();
        const uint64_t dA = sw128_desc(smem_u32(qst + st * kTileBytes), 16, 1024);
        const uint32_t tO = tmem + 64 * b;
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) umma_bf16(tO, dmove(dA, ks * 32), dmove(dHi, ks * 32), idO, ks > 0);
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) umma_bf16(tO, dmove(dA, ks * 32), dmove(dLo, ks * 32), idO, 1u);
        umma_commit(qempty + st);
        umma_commit(ofull + b);
      }
      if (!ok) *abort_flag = 1;
    }
  } else if (warp == 6) {
    if (lane == 0) {  // ------------------------------------------------ output store
      bool ok = true;
      for (int t = t0, G = 0; t < t1; ++t, ++G) {
        if (!(ok = LWAIT(staged, G & 1))) break;
        fence_proxy_async_smem();
        tma_store_5d(&to, smem_u32(ost), 0, t * kTile, 0, 0, bh);
        bulk_commit();
        bulk_wait_read();  // the staging tile may be rewritten once the store has read it
        mbar_arrive(sfree);
      }
      bulk_wait_all();
      if (!ok) *abort_flag = 1;
    }
  } else {
    // ------------------------------------------------------------------ phi, denominator, epilogue
    const int quad = warp & 3;
    const int r = quad * 32 + lane;  // tile row = TMEM lane
    const int tid = threadIdx.x - 64;
    // S^T parts into swizzled shared memory, z alongside
    for (int i = tid; i < 2 * 64 * 8; i += 128) {
      const int m = i >> 9, row = (i >> 3) & 63, c = i & 7;
      const __nv_bfloat16* src = (m ? a.stl : a.sth) + ((size_t)bh * kD + row) * kD + c * 8;
      *reinterpret_cast<uint4*>((m ? sLo : sHi) + swz(row, c)) = *reinterpret_cast<const uint4*>(src);
    }
    if (tid < kD) zs[tid] = a.zt[(size_t)bh * kD + tid];
    fence_proxy_async_smem();
    asm volatile("bar.sync 1, 128;" ::: "memory");  // z visible to all four math warps
    __syncwarp();
    if (lane == 0) mbar_arrive(sready);
    // phi of tile G + 1 runs while the tensor core computes tile G
    auto phi_tile = [&](int G, float& den) -> bool {
      const int st = G % kQStages, n = G / kQStages;
      if (!LWAIT(qfull + st, n & 1)) return false;
      uint8_t* qt = qst + st * kTileBytes;
      den = 0.f;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        uint4* p = reinterpret_cast<uint4*>(qt + swz(r, c));
        float f[8];
        *p = phi_chunk(*p, true, f);
#pragma unroll
        for (int e = 0; e < 8; ++e) den = fmaf(f[e], zs[c * 8 + e], den);
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(aready + st);
      return true;
    };
    const int count = t1 - t0;
    float den_cur = 0.f, den_next = 0.f;
    bool ok = count <= 0 || phi_tile(0, den_cur);
    for (int G = 0; G < count && ok; ++G) {
      if (G + 1 < count && !(ok = phi_tile(G + 1, den_next))) break;
      const int b = G & 1;
      if (!(ok = LWAIT(ofull + b, (G >> 1) & 1))) break;
      tc_fence_after();
      uint32_t o0[32], o1[32];
      const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + 64 * b;
      tmem_ld32(tl, o0);
      tmem_ld32(tl + 32, o1);
      tmem_wait_ld(o0);
      tmem_wait_ld(o1);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(ofree + b);
      // row r of the output tile into the staging buffer once the previous store read it
      if (G > 0 && !(ok = LWAIT(sfree, (G - 1) & 1))) break;
      const float inv = 1.f / den_cur;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint32_t* o = c < 4 ? o0 + 8 * c : o1 + 8 * (c - 4);
        *reinterpret_cast<uint4*>(ost + swz(r, c)) =
            make_uint4(pack_bf16(__uint_as_float(o[0]) * inv, __uint_as_float(o[1]) * inv),
                       pack_bf16(__uint_as_float(o[2]) * inv, __uint_as_float(o[3]) * inv),
                       pack_bf16(__uint_as_float(o[4]) * inv, __uint_as_float(o[5]) * inv),
                       pack_bf16(__uint_as_float(o[6]) * inv, __uint_as_float(o[7]) * inv));
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(staged);
      den_cur = den_next;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 128);
  }
}

// =================================================================== backward
// For the loss sum(out * g) (g = dOut) with den_i = phi(q_i) . z:
//   U_i     = S^T g_i (d-vector, u_k = sum_v S[k][v] g_i[v])
//   go_i    = phi(q_i) . U_i / den_i                      (= g_i . out_i)
//   dq_i    = (U_i - z go_i) / den_i * phi'(q_i)
//   dS      = sum_i phi(q_i) (g_i / den_i)^T,  dz = -sum_i phi(q_i) go_i / den_i
//   dk_n    = (dS v_n + dz) * phi'(k_n),       dv_n = dS^T phi(k_n)
// with phi'(x) = 1 for x > 0 and exp(x) = phi(x) otherwise, so phi' follows
// from phi alone (phi > 1 exactly when x > 0).  Three kernels, HBM-bound: a
// query pass (dq, split-N partials of dS and dz), a fixed-order compensated
// combine, and a key pass (dk, dv).  Products whose accuracy matters for the
// cancellation in dq (U) and for the N-long sums (dS) use BF16 high and low
// parts of both factors (S, phi(q), g / den), so the rounding of the tensor
// core's BF16 operands stays below 2^-16; phi(k) and dS in the key pass are
// split the same way.

// Both backward passes run two groups of eight math warps (two warps per TMEM
// lane quadrant and group) on alternating tiles: a tile's work is a chain of
// loads, exchanges and products whose latency one group cannot hide (with one
// group the passes ran at a third of the HBM rate with 2 of 16 possible warps
// per scheduler busy).
constexpr int kThreadsB = 64 + 2 * 256;      // producer, issuer, 2 x 8 math warps
constexpr int kBQStages = 3;                 // (q, g) ring; phi's and g / den's high parts replace them in place
constexpr int kBQRaw = 16384 + 5120;         // S^T hi, lo (8 KB each), z, the row-sum exchanges, padding
constexpr int kBQLo = kBQRaw + kBQStages * 2 * kTileBytes;  // per group: phi lo, g / den lo
constexpr int kBQOut = kBQLo + 2 * 2 * kTileBytes;          // staged dq, 2 KB per math warp
constexpr int kBQBar = kBQOut + 16 * 2048;
constexpr int kBQSmem = kBQBar + 1024 + 256;
constexpr int kBKStages = 4;                 // (k, v) ring; phi hi, then dk, replace k and dv replaces v in place
constexpr int kBKRaw = 32768 + 1024;         // dS hi, lo, dS^T hi, lo, then dz and padding
constexpr int kBKLo = kBKRaw + kBKStages * 2 * kTileBytes;  // per group: phi lo
constexpr int kBKBar = kBKLo + 2 * kTileBytes;
constexpr int kBKSmem = kBKBar + 1024 + 256;

// phi of two BF16 values (one 32-bit word) as an FP32 pair: max(x, 0) + min(exp x, 1)
__device__ __forceinline__ uint64_t phi_pair(uint32_t w) {
  const float x0 = __uint_as_float(w << 16), x1 = __uint_as_float(w & 0xffff0000u);
  float e0, e1;
  f2unpack(fmul2(f2pack(x0, x1), f2pack(1.4426950408889634f, 1.4426950408889634f)), e0, e1);
  return fadd2(f2pack(fmax_nan(x0, 0.f), fmax_nan(x1, 0.f)), f2pack(fmin_nan(ex2(e0), 1.f), fmin_nan(ex2(e1), 1.f)));
}
// BF16 high and low parts of an FP32 pair
__device__ __forceinline__ void split_pair(uint64_t f, uint32_t& hi, uint32_t& lo) {
  float a, b;
  f2unpack(f, a, b);
  hi = pack_bf16(a, b);
  f2unpack(ffma2(u2pack(hi << 16, hi & 0xffff0000u), f2pack(-1.f, -1.f), f), a, b);
  lo = pack_bf16(a, b);
}

// 64 x 64 BF16 matrices (rows of 128 bytes) from global memory into 128-byte-
// swizzled shared memory, n of them; every math thread (tid 0..nthr - 1) takes part
__device__ __forceinline__ void load_mats(int tid, int nthr, int n, const __nv_bfloat16* const* src,
                                          uint8_t* const* dst) {
  for (int i = tid; i < n * 64 * 8; i += nthr) {
    const int m = i >> 9, row = (i >> 3) & 63, c = i & 7;
    *reinterpret_cast<uint4*>(dst[m] + swz(row, c)) = *reinterpret_cast<const uint4*>(src[m] + row * kD + c * 8);
  }
}

struct BQArgs {
  int N, BH, ntiles, chunk_tiles, sum_tiles;
  const __nv_bfloat16* sth;  // forward summary S^T, high and low parts [BH, 64 (v), 64 (k)]
  const __nv_bfloat16* stl;
  const float* zt;           // [BH, 64]
  float* part_dS;            // [chunks, BH, 64 (k), 64 (v)]
  float* part_dz;            // [chunks, BH, 64]
};

// Query pass, grid (chunks, BH): every CTA streams a chunk of 128-token query
// tiles (q and g by TMA through three stages), tile t going to math group t & 1.
//   issuer: U = G S (A = g tile K-major, B = S^T parts MN-major), into the
//           group's TMEM buffer, two tiles ahead; dS += phi(Q)^T (G / den) over
//           the tile's 128 tokens (both operands MN-major; chains hi.hi, hi.lo,
//           lo.hi)
//   math:   per row, phi(q) and den in FP32, phi's parts over the q tile and in
//           the group's low tile; with U: go, dq (staged per warp, stored by
//           TMA, which also drops rows past N), dz; g / den's parts over the g
//           tile and in the low tile.  The two warps of a lane quadrant take 32
//           of a row's 64 columns each and exchange the row's two sums (den,
//           phi(q) . U) through shared memory, added in a fixed order.
// At the end the CTA writes its dS and dz partials.  16 heads of 262144
// tokens: 705 -> 453 us (one group of eight warps, plain stores of dq and
// 1216 CTAs before; 436 without the folds); 1.61 GB, 0.53 of the HBM rate: the math
// groups' row work (phi, its parts, the row sums) sets the pace.
__global__ void __launch_bounds__(kThreadsB, 1) la_bwd_query_kernel(const __grid_constant__ CUtensorMap tq,
                                                                    const __grid_constant__ CUtensorMap tg,
                                                                    const __grid_constant__ CUtensorMap tdq,
                                                                    const BQArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sHi = smem;
  uint8_t* sLo = smem + 8192;
  float* zs = reinterpret_cast<float*>(smem + 16384);
  float* xsum = reinterpret_cast<float*>(smem + 16384 + 256);  // [group][den, go][half][128 rows]
  auto stq = [&](int st) { return smem + kBQRaw + st * 2 * kTileBytes; };  // q, then phi hi
  auto stg = [&](int st) { return stq(st) + kTileBytes; };                 // g, then g/den hi
  auto lop = [&](int grp) { return smem + kBQLo + grp * 2 * kTileBytes; };  // phi lo
  auto glo = [&](int grp) { return lop(grp) + kTileBytes; };                // g/den lo
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kBQBar);
  uint64_t* empty = full + kBQStages;
  uint64_t* ufull = empty + kBQStages;  // [group]
  uint64_t* ufree = ufull + 2;          // [group]
  uint64_t* dsready = ufree + 2;        // [group]
  uint64_t* lofree = dsready + 2;       // [group]
  uint64_t* sfull = lofree + 2;         // [2]: a dS accumulator's last product is complete
  uint64_t* sfree = sfull + 2;          // [2]: it has been folded
  uint64_t* sready = sfree + 2;
  uint64_t* done = sready + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = blockIdx.x, bh = blockIdx.y;
  const int t0 = chunk * a.chunk_tiles, t1 = min(a.ntiles, t0 + a.chunk_tiles);
  const int count = t1 - t0;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kBQStages; ++i) {
      mbar_init(full + i, 1);
      mbar_init(empty + i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(ufull + i, 1);
      mbar_init(ufree + i, 8);
      mbar_init(dsready + i, 8);
      mbar_init(lofree + i, 1);
      mbar_init(sfull + i, 1);
      mbar_init(sfree + i, 8);
    }
    mbar_init(sready, 16);
    mbar_init(done, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tq);
    prefetch_tmap(&tg);
    prefetch_tmap(&tdq);
  }
  if (warp == 1) {
    // the groups' U buffers at columns 0 and 64, dS accumulators (M = 64) at 128 and 192, their sum at 256, its
    // compensation at 320
    tmem_alloc(tslot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {  // ------------------------------------------------ TMA producer
      uint32_t armed = 0, par = 0;
      bool ok = true;
      for (int G = 0; G < count; ++G) {
        const int st = G % kBQStages, n = G / kBQStages;
        if (!(ok = LWAIT(empty + st, (n & 1) ^ 1))) break;
        mbar_arrive_expect_tx(full + st, 2 * kTileBytes);
        armed |= 1u << st;
        par = (par & ~(1u << st)) | ((n & 1) << st);
        tma_load_5d(stq(st), &tq, full + st, 0, (t0 + G) * kTile, 0, 0, bh);
        tma_load_5d(stg(st), &tg, full + st, 0, (t0 + G) * kTile, 0, 0, bh);
      }
      if (!ok)
        for (int s2 = 0; s2 < kBQStages; ++s2)
          if (armed & (1u << s2)) mbar_wait<set_status_l>(full + s2, (par >> s2) & 1, abort_flag, false);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ------------------------------------------------ MMA issuer
      constexpr uint32_t idU = idesc_bf16(128, 64, 1);                 // B = S^T rows, MN-major
      constexpr uint32_t idDS = idesc_bf16(64, 64, 1) | (1u << 15);    // A and B MN-major
      const uint64_t dSh = sw128_desc(smem_u32(sHi), 16384, 1024), dSl = sw128_desc(smem_u32(sLo), 16384, 1024);
      bool ok = LWAIT(sready, 0);
      // U of tile G into its group's buffer
      auto issue_u = [&](int G) -> bool {
        const int st = G % kBQStages, b = G & 1;
        if (!LWAIT(full + st, (G / kBQStages) & 1)) return false;
        if (G >= 2 && !LWAIT(ufree + b, ((G >> 1) - 1) & 1)) return false;
        tc_fence_after();
        const uint32_t tU = tmem + 64 * b;
        const uint64_t dG = sw128_desc(smem_u32(stg(st)), 16, 1024);
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) umma_bf16(tU, dmove(dG, ks * 32), dmove(dSh, ks * 2048), idU, ks > 0);
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) umma_bf16(tU, dmove(dG, ks * 32), dmove(dSl, ks * 2048), idU, 1u);
        umma_commit(ufull + b);
        return true;
      };
      for (int G = 0; G < 2 && G < count && ok; ++G) ok = issue_u(G);
      int m = 0, ch = 0;  // tile within its sum, sum
      for (int G = 0; G < count && ok; ++G) {
        const int st = G % kBQStages, b = G & 1, sb = ch & 1;
        // dS += phi(Q)^T (G / den) once the math warps wrote both operands' parts
        if (!(ok = LWAIT(dsready + b, (G >> 1) & 1))) break;
        if (m == 0 && ch >= 2 && !(ok = LWAIT(sfree + sb, ((ch >> 1) - 1) & 1))) break;
        tc_fence_after();
        const uint32_t tD = tmem + 128 + 64 * sb;
        const uint64_t pH = sw128_desc(smem_u32(stq(st)), 16384, 1024), pL = sw128_desc(smem_u32(lop(b)), 16384, 1024);
        const uint64_t gH = sw128_desc(smem_u32(stg(st)), 16384, 1024), gL = sw128_desc(smem_u32(glo(b)), 16384, 1024);
#pragma unroll
        for (int ks = 0; ks < kTile / 16; ++ks)
          umma_bf16(tD, dmove(pH, ks * 2048), dmove(gH, ks * 2048), idDS, (m > 0 || ks > 0) ? 1u : 0u);
#pragma unroll
        for (int ks = 0; ks < kTile / 16; ++ks) umma_bf16(tD, dmove(pH, ks * 2048), dmove(gL, ks * 2048), idDS, 1u);
#pragma unroll
        for (int ks = 0; ks < kTile / 16; ++ks) umma_bf16(tD, dmove(pL, ks * 2048), dmove(gH, ks * 2048), idDS, 1u);
        umma_commit(empty + st);
        umma_commit(lofree + b);
        if (++m == a.sum_tiles) {
          umma_commit(sfull + sb);
          m = 0;
          ++ch;
        }
        if (G + 2 < count) ok = issue_u(G + 2);
      }
      umma_commit(done);
      if (!ok) *abort_flag = 1;
      mbar_wait<set_status_l>(done, 0, abort_flag, false);  // before tensor memory is released
    }
  } else {
    // ------------------------------------------------------------------ math warps
    const int quad = warp & 3;
    const int grp = (warp - 2) >> 3;
    const int h = ((warp - 2) >> 2) & 1;  // columns [32 h, 32 h + 32) of the row: chunks 4 h .. 4 h + 3
    const int r = quad * 32 + lane;       // tile row = TMEM lane
    const int tid = threadIdx.x - 64;
    const int pair_bar = 2 + grp * 4 + quad;  // named barrier of the two warps of this group and lane quadrant
    {
      const __nv_bfloat16* src[2] = {a.sth + (size_t)bh * kD * kD, a.stl + (size_t)bh * kD * kD};
      uint8_t* dst[2] = {sHi, sLo};
      load_mats(tid, 512, 2, src, dst);
      if (tid < kD) zs[tid] = a.zt[(size_t)bh * kD + tid];
      fence_proxy_async_smem();
      asm volatile("bar.sync 1, 512;" ::: "memory");  // z visible to all math warps
      __syncwarp();
      if (lane == 0) mbar_arrive(sready);
    }
    const uint32_t zaddr = smem_u32(zs) + h * 128;
    float* xden = xsum + grp * 512;
    float* xgo = xden + 256;
    const uint32_t out = smem_u32(smem + kBQOut) + (warp - 2) * 2048;  // 32 rows x 64 bytes, 64-byte swizzle
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + 64 * grp + 32 * h;
    uint64_t dz[kD / 4];
#pragma unroll
    for (int i = 0; i < kD / 4; ++i) dz[i] = 0;
    // group 0 folds the sums of dS, `ch` of them so far
    const uint32_t ts = tl + 128;
    int ch = 0;
    auto fold = [&]() -> bool {
      if (!WARP_LWAIT(sfull + (ch & 1), (ch >> 1) & 1)) return false;
      tc_fence_after();
      fold_sum(ts + 64 * (ch & 1), ts + 128, ts + 192, ch == 0);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(sfree + (ch & 1));
      ++ch;
      return true;
    };
    bool ok = true;
    for (int G = grp, n = 0; G < count; G += 2, ++n) {
      const int st = G % kBQStages;
      const bool valid = (int64_t)(t0 + G) * kTile + r < a.N;
      // (a failed wait is carried to the pair's next vote: what is computed until
      // then stays in shared memory)
      ok = ok && WARP_LWAIT(full + st, (G / kBQStages) & 1);
      // the group's low tiles are free once its previous tile's dS product is done
      if (n > 0) ok = ok && WARP_LWAIT(lofree + grp, (n - 1) & 1);
      // phi(q) in FP32, this half's part of den, and phi's parts (hi over q, lo in the low tile)
      const uint32_t aq = smem_u32(stq(st)), ap = smem_u32(lop(grp));
      uint64_t dp2 = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t off = swz(r, 4 * h + c);
        const uint4 u = ld_shared_v4(aq + off), za = ld_shared_v4(zaddr + c * 32), zb = ld_shared_v4(zaddr + c * 32 + 16);
        const uint64_t f0 = phi_pair(u.x), f1 = phi_pair(u.y), f2 = phi_pair(u.z), f3 = phi_pair(u.w);
        dp2 = ffma2(f0, u2pack(za.x, za.y), dp2);
        dp2 = ffma2(f1, u2pack(za.z, za.w), dp2);
        dp2 = ffma2(f2, u2pack(zb.x, zb.y), dp2);
        dp2 = ffma2(f3, u2pack(zb.z, zb.w), dp2);
        uint32_t hi[4], lo[4];
        split_pair(f0, hi[0], lo[0]);
        split_pair(f1, hi[1], lo[1]);
        split_pair(f2, hi[2], lo[2]);
        split_pair(f3, hi[3], lo[3]);
        st_shared_v4(aq + off, hi[0], hi[1], hi[2], hi[3]);
        st_shared_v4(ap + off, lo[0], lo[1], lo[2], lo[3]);
      }
      float d0, d1;
      f2unpack(dp2, d0, d1);
      xden[h * 128 + r] = d0 + d1;
      if (!(ok = pair_vote(pair_bar, ok))) break;
      const float den = xden[r] + xden[128 + r];
      const float inv = valid ? 1.f / den : 0.f;
      // this half of the U row (the U product is done: the g tile may be overwritten below)
      ok = WARP_LWAIT(ufull + grp, n & 1);
      tc_fence_after();
      // phi(q) again from its parts, eight columns of a chunk at a time
      auto phi_parts = [&](int c, uint64_t (&f)[4]) {
        const uint32_t off = swz(r, 4 * h + c);
        const uint4 hi = ld_shared_v4(aq + off), lo = ld_shared_v4(ap + off);
        f[0] = fadd2(u2pack(hi.x << 16, hi.x & 0xffff0000u), u2pack(lo.x << 16, lo.x & 0xffff0000u));
        f[1] = fadd2(u2pack(hi.y << 16, hi.y & 0xffff0000u), u2pack(lo.y << 16, lo.y & 0xffff0000u));
        f[2] = fadd2(u2pack(hi.z << 16, hi.z & 0xffff0000u), u2pack(lo.z << 16, lo.z & 0xffff0000u));
        f[3] = fadd2(u2pack(hi.w << 16, hi.w & 0xffff0000u), u2pack(lo.w << 16, lo.w & 0xffff0000u));
      };
      uint64_t gp2 = 0;
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        uint32_t u[16];
        tmem_ld16(tl + 16 * hh, u);
        tmem_wait_ld(u);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint64_t f[4];
          phi_parts(2 * hh + c, f);
#pragma unroll
          for (int e = 0; e < 4; ++e) gp2 = ffma2(f[e], u2pack(u[8 * c + 2 * e], u[8 * c + 2 * e + 1]), gp2);
        }
      }
      f2unpack(gp2, d0, d1);
      xgo[h * 128 + r] = d0 + d1;
      if (lane == 0) bulk_wait_read();  // the previous dq store has read this warp's staging block
      if (!(ok = pair_vote(pair_bar, ok))) break;
      const float go = (xgo[r] + xgo[128 + r]) * inv;
      // dq = (U - z go) / den * phi'(q); dz -= phi(q) go / den
      const uint64_t ngo2 = f2pack(-go, -go), inv2 = f2pack(inv, inv), ngi2 = f2pack(-(go * inv), -(go * inv));
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        uint32_t u[16];
        tmem_ld16(tl + 16 * hh, u);
        tmem_wait_ld(u);
        if (hh == 1) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(ufree + grp);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int cc = 2 * hh + c;
          uint64_t f[4];
          phi_parts(cc, f);
          const uint4 za = ld_shared_v4(zaddr + cc * 32), zb = ld_shared_v4(zaddr + cc * 32 + 16);
          const uint64_t z[4] = {u2pack(za.x, za.y), u2pack(za.z, za.w), u2pack(zb.x, zb.y), u2pack(zb.z, zb.w)};
          uint32_t pk[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float f0, f1;
            f2unpack(f[e], f0, f1);
            const uint64_t t = fmul2(ffma2(z[e], ngo2, u2pack(u[8 * c + 2 * e], u[8 * c + 2 * e + 1])), inv2);
            f2unpack(fmul2(t, f2pack(fmin_nan(f0, 1.f), fmin_nan(f1, 1.f))), f0, f1);
            pk[e] = pack_bf16(f0, f1);
            dz[4 * cc + e] = ffma2(f[e], ngi2, dz[4 * cc + e]);
          }
          st_shared_v4(out + lane * 64 + ((cc ^ ((lane >> 1) & 3)) << 4), pk[0], pk[1], pk[2], pk[3]);
        }
      }
      // g / den: hi over the g tile, lo in the low tile
      const uint32_t ag = smem_u32(stg(st)), al = smem_u32(glo(grp));
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t off = swz(r, 4 * h + c);
        const uint4 u = ld_shared_v4(ag + off);
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) split_pair(fmul2(u2pack(w[e] << 16, w[e] & 0xffff0000u), inv2), hi[e], lo[e]);
        st_shared_v4(ag + off, hi[0], hi[1], hi[2], hi[3]);
        st_shared_v4(al + off, lo[0], lo[1], lo[2], lo[3]);
      }
      fence_proxy_async_smem();  // the tensor core and the copy unit read what these threads wrote
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(dsready + grp);
        tma_store_5d(&tdq, out, 32 * h, (t0 + G) * kTile + quad * 32, 0, 0, bh);
        bulk_commit();
      }
      if (grp == 0)  // sums that ended before this tile
        while (ok && (ch + 1) * a.sum_tiles <= G) ok = fold();
    }
    if (grp == 0)
      while (ok && (ch + 1) * a.sum_tiles < count) ok = fold();
    // epilogue: dS partial (M = 64: rows 16q .. 16q+15 in lanes 0..15 of lane
    // quadrant q; group 0's warps, 32 of the 64 columns each) and dz reduced
    // over both groups' 128 rows in fixed order
    const bool got = ok && WARP_LWAIT(done, 0);
    tc_fence_after();
    const size_t part = (size_t)chunk * a.BH + bh;
    if (grp == 0) {
      uint32_t s0[32];
      last_sum(ts + 64 * (ch & 1), ts + 128, ts + 192, ch == 0, s0);
      if (got && lane < 16) {
        float* dst = a.part_dS + (part * kD + quad * 16 + lane) * kD + 32 * h;
#pragma unroll
        for (int j = 0; j < 32; j += 4)
          *reinterpret_cast<float4*>(dst + j) = make_float4(__uint_as_float(s0[j]), __uint_as_float(s0[j + 1]),
                                                            __uint_as_float(s0[j + 2]), __uint_as_float(s0[j + 3]));
      }
    }
    // the low tiles are idle once `done` completed: reuse them for the dz rows
    float* zbuf = reinterpret_cast<float*>(smem + kBQLo);
    if (got) {
#pragma unroll
      for (int i = 0; i < kD / 4; ++i) {
        float x, y;
        f2unpack(dz[i], x, y);
        *reinterpret_cast<float2*>(zbuf + (grp * kTile + r) * kD + 32 * h + 2 * i) = make_float2(x, y);
      }
    }
    const float sum = column_sum<512, 2 * kTile>(zbuf, tid);
    if (got && tid < kD) a.part_dz[part * kD + tid] = sum;
    if (lane == 0) bulk_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

struct BCombArgs {
  int BH, chunks;
  const float* part_dS;
  const float* part_dz;
  __nv_bfloat16 *dsh, *dsl;    // dS [BH, 64 (k), 64 (v)], high and low parts
  __nv_bfloat16 *dsth, *dstl;  // dS^T [BH, 64 (v), 64 (k)]
  float* dz;                   // [BH, 64]
};

// grid (BH, ceil((64 * 64 + 64) / 256)): one entry per thread, chunk
// partials summed in ascending chunk order with Kahan compensation
__global__ void __launch_bounds__(256) la_bwd_combine_kernel(const BCombArgs a) {
  const int bh = blockIdx.x;
  for (int e = blockIdx.y * 256 + threadIdx.x; e < kD * kD + kD; e += 256 * gridDim.y) {
    const bool is_z = e >= kD * kD;
    float sum = 0.f, comp = 0.f;
    const float* src = is_z ? a.part_dz + (size_t)bh * kD + (e - kD * kD) : a.part_dS + (size_t)bh * kD * kD + e;
    kahan_chunks(src, (size_t)a.BH * (is_z ? kD : kD * kD), a.chunks, sum, comp);
    if (is_z) {
      a.dz[(size_t)bh * kD + (e - kD * kD)] = sum;
    } else {
      const int k = e / kD, v = e % kD;
      const __nv_bfloat16 hi = __float2bfloat16_rn(sum);
      const __nv_bfloat16 lo = __float2bfloat16_rn(sum - __bfloat162float(hi));
      const size_t m = (size_t)bh * kD * kD;
      a.dsh[m + k * kD + v] = hi;
      a.dsl[m + k * kD + v] = lo;
      a.dsth[m + v * kD + k] = hi;
      a.dstl[m + v * kD + k] = lo;
    }
  }
}

struct BKArgs {
  int ntiles, tiles_per_cta;
  const __nv_bfloat16 *dsh, *dsl, *dsth, *dstl;
  const float* dz;
};

// Key pass, grid (ceil(ntiles / tiles_per_cta), BH): per 128-token key tile
// (k and v by TMA through four stages), tile t going to math group t & 1
//   math:   phi(k)'s parts (hi over the k tile, lo in the group's low tile)
//   issuer: P1 = V dS^T (A = v tile, B = dS rows; hi and lo) and P2 = phi(K) dS
//           (A = phi parts, B = dS^T rows; chains hi.hi, hi.lo, lo.hi), into
//           the group's TMEM buffers
//   math:   dk = (P1 + dz) * phi'(k) over the k tile, dv = P2 over the v tile
//           (the products have read both), 32 rows of each stored by TMA per
//           lane quadrant (rows past N are dropped)
// A stage is released by the four quadrants once their stores have read it.
// Two math warps per group and TMEM lane quadrant, each taking 32 of a row's
// 64 columns (nothing here sums over a row).  16 heads of 262144 tokens:
// 713 -> 324 us (one group of eight warps, a thread storing its own 64
// bytes of a row and 16 tiles per CTA before); 2.15 GB in that time, 0.98 of
// the HBM rate.
__global__ void __launch_bounds__(kThreadsB, 1) la_bwd_key_kernel(const __grid_constant__ CUtensorMap tk,
                                                                  const __grid_constant__ CUtensorMap tv,
                                                                  const __grid_constant__ CUtensorMap tdk,
                                                                  const __grid_constant__ CUtensorMap tdv,
                                                                  const BKArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* mDh = smem;          // dS rows (k), hi
  uint8_t* mDl = smem + 8192;   // dS rows, lo
  uint8_t* mTh = smem + 16384;  // dS^T rows (v), hi
  uint8_t* mTl = smem + 24576;  // dS^T rows, lo
  float* dzs = reinterpret_cast<float*>(smem + 32768);
  auto stk = [&](int st) { return smem + kBKRaw + st * 2 * kTileBytes; };  // k, then phi hi, then dk
  auto stv = [&](int st) { return stk(st) + kTileBytes; };                 // v, then dv
  auto lop = [&](int grp) { return smem + kBKLo + grp * kTileBytes; };     // phi lo
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kBKBar);
  uint64_t* empty = full + kBKStages;
  uint64_t* kready = empty + kBKStages;  // [group]
  uint64_t* pfull = kready + 2;          // [group]
  uint64_t* pfree = pfull + 2;           // [group]
  uint64_t* sready = pfree + 2;
  uint64_t* done = sready + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bh = blockIdx.y;
  const int t0 = blockIdx.x * a.tiles_per_cta, t1 = min(a.ntiles, t0 + a.tiles_per_cta);
  const int count = t1 - t0;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kBKStages; ++i) {
      mbar_init(full + i, 1);
      mbar_init(empty + i, 4);  // the lane quadrants of the tile's group
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(kready + i, 8);
      mbar_init(pfull + i, 1);
      mbar_init(pfree + i, 8);
    }
    mbar_init(sready, 16);
    mbar_init(done, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tk);
    prefetch_tmap(&tv);
    prefetch_tmap(&tdk);
    prefetch_tmap(&tdv);
  }
  if (warp == 1) {
    tmem_alloc(tslot, 256);  // group b: P1 at 128 b, P2 at 128 b + 64
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  if (warp == 0) {
    if (lane == 0) {  // ------------------------------------------------ TMA producer
      uint32_t armed = 0, par = 0;
      bool ok = true;
      for (int G = 0; G < count; ++G) {
        const int st = G % kBKStages, n = G / kBKStages;
        if (!(ok = LWAIT(empty + st, (n & 1) ^ 1))) break;
        mbar_arrive_expect_tx(full + st, 2 * kTileBytes);
        armed |= 1u << st;
        par = (par & ~(1u << st)) | ((n & 1) << st);
        tma_load_5d(stk(st), &tk, full + st, 0, (t0 + G) * kTile, 0, 0, bh);
        tma_load_5d(stv(st), &tv, full + st, 0, (t0 + G) * kTile, 0, 0, bh);
      }
      if (!ok)
        for (int s2 = 0; s2 < kBKStages; ++s2)
          if (armed & (1u << s2)) mbar_wait<set_status_l>(full + s2, (par >> s2) & 1, abort_flag, false);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ------------------------------------------------ MMA issuer
      constexpr uint32_t idP = idesc_bf16(128, 64, 0);  // A, B K-major
      const uint64_t bDh = sw128_desc(smem_u32(mDh), 16, 1024), bDl = sw128_desc(smem_u32(mDl), 16, 1024);
      const uint64_t bTh = sw128_desc(smem_u32(mTh), 16, 1024), bTl = sw128_desc(smem_u32(mTl), 16, 1024);
      bool ok = LWAIT(sready, 0);
      for (int G = 0; G < count && ok; ++G) {
        const int st = G % kBKStages, b = G & 1;
        if (!(ok = LWAIT(full + st, (G / kBKStages) & 1))) break;
        if (G >= 2 && !(ok = LWAIT(pfree + b, ((G >> 1) - 1) & 1))) break;
        tc_fence_after();
        const uint32_t tP1 = tmem + 128 * b, tP2 = tP1 + 64;
        const uint64_t aV = sw128_desc(smem_u32(stv(st)), 16, 1024);
        const uint64_t aH = sw128_desc(smem_u32(stk(st)), 16, 1024), aL = sw128_desc(smem_u32(lop(b)), 16, 1024);
        // P1 needs only v: it runs while phi is formed
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) umma_bf16(tP1, dmove(aV, ks * 32), dmove(bDh, ks * 32), idP, ks > 0);
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) umma_bf16(tP1, dmove(aV, ks * 32), dmove(bDl, ks * 32), idP, 1u);
        if (!(ok = LWAIT(kready + b, (G >> 1) & 1))) break;
        tc_fence_after();
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) umma_bf16(tP2, dmove(aH, ks * 32), dmove(bTh, ks * 32), idP, ks > 0);
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) umma_bf16(tP2, dmove(aH, ks * 32), dmove(bTl, ks * 32), idP, 1u);
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) umma_bf16(tP2, dmove(aL, ks * 32), dmove(bTh, ks * 32), idP, 1u);
        umma_commit(pfull + b);
      }
      umma_commit(done);
      if (!ok) *abort_flag = 1;
      mbar_wait<set_status_l>(done, 0, abort_flag, false);  // before tensor memory is released
    }
  } else {
    // ------------------------------------------------------------------ math warps
    const int quad = warp & 3;
    const int grp = (warp - 2) >> 3;
    const int h = ((warp - 2) >> 2) & 1;  // columns [32 h, 32 h + 32) of the row: chunks 4 h .. 4 h + 3
    const int r = quad * 32 + lane;
    const int tid = threadIdx.x - 64;
    const int pair_bar = 2 + grp * 4 + quad;  // named barrier of the two warps of this group and lane quadrant
    {
      const size_t m = (size_t)bh * kD * kD;
      const __nv_bfloat16* src[4] = {a.dsh + m, a.dsl + m, a.dsth + m, a.dstl + m};
      uint8_t* dst[4] = {mDh, mDl, mTh, mTl};
      load_mats(tid, 512, 4, src, dst);
      if (tid < kD) dzs[tid] = a.dz[(size_t)bh * kD + tid];
      fence_proxy_async_smem();
      asm volatile("bar.sync 1, 512;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(sready);
    }
    const uint32_t zaddr = smem_u32(dzs) + h * 128;
    const uint32_t al = smem_u32(lop(grp));
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16) + 128 * grp + 32 * h;
    const bool storer = h == 0 && lane == 0;  // stores its quadrant's rows
    bool ok = true;
    for (int G = grp, n = 0; G < count; G += 2, ++n) {
      const int st = G % kBKStages;
      if (n > 0 && storer) {  // the previous tile's stores have read their stage
        bulk_wait_read();
        mbar_arrive(empty + (G - 2) % kBKStages);
      }
      ok = WARP_LWAIT(full + st, (G / kBKStages) & 1);  // a failed wait is carried to the pair's vote
      const uint32_t ak = smem_u32(stk(st)), av = smem_u32(stv(st));
      uint64_t f[16];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t off = swz(r, 4 * h + c);
        const uint4 u = ld_shared_v4(ak + off);
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          f[4 * c + e] = phi_pair(w[e]);
          split_pair(f[4 * c + e], hi[e], lo[e]);
        }
        st_shared_v4(ak + off, hi[0], hi[1], hi[2], hi[3]);
        st_shared_v4(al + off, lo[0], lo[1], lo[2], lo[3]);
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(kready + grp);
      ok = ok && WARP_LWAIT(pfull + grp, n & 1);
      tc_fence_after();
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        uint32_t p1[16], p2[16];
        tmem_ld16(tl + 16 * hh, p1);
        tmem_ld16(tl + 64 + 16 * hh, p2);
        tmem_wait_ld(p1);
        tmem_wait_ld(p2);
        if (hh == 1) {
          tc_fence_before();
          __syncwarp();
          if (ok && lane == 0) mbar_arrive(pfree + grp);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int cc = 2 * hh + c;
          const uint4 za = ld_shared_v4(zaddr + cc * 32), zb = ld_shared_v4(zaddr + cc * 32 + 16);
          const uint64_t z[4] = {u2pack(za.x, za.y), u2pack(za.z, za.w), u2pack(zb.x, zb.y), u2pack(zb.z, zb.w)};
          uint32_t ok4[4], ov4[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float f0, f1;
            f2unpack(f[4 * cc + e], f0, f1);
            const uint64_t t = fadd2(u2pack(p1[8 * c + 2 * e], p1[8 * c + 2 * e + 1]), z[e]);
            f2unpack(fmul2(t, f2pack(fmin_nan(f0, 1.f), fmin_nan(f1, 1.f))), f0, f1);
            ok4[e] = pack_bf16(f0, f1);
            ov4[e] = pack_bf16(__uint_as_float(p2[8 * c + 2 * e]), __uint_as_float(p2[8 * c + 2 * e + 1]));
          }
          const uint32_t off = swz(r, 4 * h + cc);
          st_shared_v4(ak + off, ok4[0], ok4[1], ok4[2], ok4[3]);
          st_shared_v4(av + off, ov4[0], ov4[1], ov4[2], ov4[3]);
        }
      }
      fence_proxy_async_smem();  // the copy unit reads what these threads wrote
      if (!(ok = pair_vote(pair_bar, ok))) break;
      if (storer) {
        tma_store_5d(&tdk, ak + quad * 4096, 0, (t0 + G) * kTile + quad * 32, 0, 0, bh);
        tma_store_5d(&tdv, av + quad * 4096, 0, (t0 + G) * kTile + quad * 32, 0, 0, bh);
        bulk_commit();
      }
    }
    if (storer) bulk_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
}

constexpr int kSumSmem = kStagesS * kSumStage + 1024 + 256;
constexpr int kQSmem = 16384 + (kQStages + 1) * kTileBytes + 1024 + 512;

}  // namespace

// Tiles per CTA for BH heads of `ntiles` tiles on `slots` resident CTAs: the
// fewest waves (up to four) that leave at most 5 % of the slots empty, else the
// fullest.  Every CTA pays for its tensor memory, its operand matrices and the
// fill of its ring, and the split-N passes for a partial that the combine reads
// (forward and backward, one head of 1.5 M tokens: 1087 -> 484 us with the
// sixteen-load combine, half of it from the combines; 16 heads of 262144:
// 1360 -> 1164, 1183 with the folded sums; before, 1216 CTAs or 16 tiles each
// whatever the problem).
static int tiles_per_cta(int ntiles, int BH, int slots) {
  int best = 1;
  double full = 0.0;
  for (int w = 1; w <= 4; ++w) {
    const int want = slots * w / BH;  // CTAs per head
    const int per = want < 1 ? ntiles : (ntiles + want - 1) / want;
    const int ctas = (ntiles + per - 1) / per * BH;
    const double f = (double)ntiles * BH / ((double)per * slots * ((ctas + slots - 1) / slots));
    if (f > full + 1e-9) {
      full = f;
      best = per;
    }
    if (full >= 0.95 || per == 1) break;  // one tile each: more waves change nothing
  }
  return best;
}

LinearPlan linear_plan(int B, int nh, int64_t N) {
  LinearPlan p;
  const int BH = B * nh;
  p.ntiles = (int)((N + kTile - 1) / kTile);
  p.chunk_tiles = tiles_per_cta(p.ntiles, BH, 304);  // two CTAs per SM
  p.chunks = (p.ntiles + p.chunk_tiles - 1) / p.chunk_tiles;
  p.q_tiles = tiles_per_cta(p.ntiles, BH, 456);      // three
  p.b_chunk_tiles = tiles_per_cta(p.ntiles, BH, 152);  // one, as the key pass
  p.b_chunks = (p.ntiles + p.b_chunk_tiles - 1) / p.b_chunk_tiles;
  // half of a CTA's share if there were 1216 CTAs (a share of two whole: a fold per
  // tile cost 4 x 60000 tokens 2 %), 16 at most
  const int share = (int)(((int64_t)p.ntiles * BH + 1215) / 1216);
  p.sum_tiles = share <= 2 ? share : share < 32 ? (share + 1) / 2 : 16;
  return p;
}

static LinearLayout layout_of(const LinearPlan& p, size_t BH) {
  LinearLayout l;
  l.part_S = 0;
  l.part_z = l.part_S + align_up((size_t)p.chunks * BH * kD * kD * 4);
  l.sth = l.part_z + align_up((size_t)p.chunks * BH * kD * 4);
  l.stl = l.sth + align_up(BH * kD * kD * 2);
  l.z = l.stl + align_up(BH * kD * kD * 2);
  l.bytes = l.z + align_up(BH * kD * 4);
  return l;
}

LinearLayout linear_layout(int B, int nh, int64_t N) {
  return layout_of(linear_plan(B, nh, N), (size_t)B * nh);
}

size_t linear_ws_bytes(int B, int nh, int64_t N) { return linear_layout(B, nh, N).bytes; }

cudaError_t launch_linear(const void* q, const void* k, const void* v, void* out, void* ws, int B, int nh, int64_t N,
                          cudaStream_t st) {
  const LinearPlan p = linear_plan(B, nh, N);
  const int BH = B * nh;
  const LinearLayout lay = layout_of(p, BH);
  char* w = static_cast<char*>(ws);
  SumArgs sa;
  sa.N = (int)N;
  sa.BH = BH;
  sa.ntiles = p.ntiles;
  sa.chunk_tiles = p.chunk_tiles;
  sa.sum_tiles = p.sum_tiles;
  sa.ws_S = reinterpret_cast<float*>(w + lay.part_S);
  sa.ws_z = reinterpret_cast<float*>(w + lay.part_z);
  CombArgs ca;
  ca.BH = BH;
  ca.chunks = p.chunks;
  ca.ws_S = sa.ws_S;
  ca.ws_z = sa.ws_z;
  ca.sth = reinterpret_cast<__nv_bfloat16*>(w + lay.sth);
  ca.stl = reinterpret_cast<__nv_bfloat16*>(w + lay.stl);
  ca.zt = reinterpret_cast<float*>(w + lay.z);
  QArgs qa;
  qa.N = (int)N;
  qa.BH = BH;
  qa.ntiles = p.ntiles;
  qa.tiles_per_cta = p.q_tiles;
  qa.sth = ca.sth;
  qa.stl = ca.stl;
  qa.zt = ca.zt;

  CUtensorMap mq, mk, mv, mo;
  if (!make_tmap_5d(&mq, q, kD, (int)N, 1, 1, BH, kTile, 1, 1) || !make_tmap_5d(&mo, out, kD, (int)N, 1, 1, BH, kTile, 1, 1) ||
      !make_tmap_5d(&mk, k, kD, (int)N, 1, 1, BH, kTile, 1, 1) || !make_tmap_5d(&mv, v, kD, (int)N, 1, 1, BH, kTile, 1, 1))
    return cudaErrorInvalidValue;
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(la_summary_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSumSmem) != cudaSuccess ||
        cudaFuncSetAttribute(la_query_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kQSmem) != cudaSuccess)
      return cudaErrorInvalidValue;
    attr = true;
  }
  prof_begin(kKLinearSummary, st);
  la_summary_kernel<<<dim3(p.chunks, BH), kThreadsL, kSumSmem, st>>>(mk, mv, sa);
  cudaError_t e = cudaGetLastError();
  prof_end(kKLinearSummary, st);
  if (e != cudaSuccess) return e;
  prof_begin(kKLinearCombine, st);
  la_combine_kernel<<<dim3(BH, (kD * kD + kD + 255) / 256), 256, 0, st>>>(ca);
  e = cudaGetLastError();
  prof_end(kKLinearCombine, st);
  if (e != cudaSuccess) return e;
  prof_begin(kKLinearQuery, st);
  la_query_kernel<<<dim3((p.ntiles + p.q_tiles - 1) / p.q_tiles, BH), kThreadsQ, kQSmem, st>>>(mq, mo,
                                                                                                             qa);
  e = cudaGetLastError();
  prof_end(kKLinearQuery, st);
  return e;
}

static LinearBwdLayout bwd_layout_of(const LinearPlan& p, size_t BH) {
  LinearBwdLayout l;
  l.part_dS = 0;
  l.part_dz = l.part_dS + align_up((size_t)p.b_chunks * BH * kD * kD * 4);
  l.dsh = l.part_dz + align_up((size_t)p.b_chunks * BH * kD * 4);
  l.dsl = l.dsh + align_up(BH * kD * kD * 2);
  l.dsth = l.dsl + align_up(BH * kD * kD * 2);
  l.dstl = l.dsth + align_up(BH * kD * kD * 2);
  l.dz = l.dstl + align_up(BH * kD * kD * 2);
  l.bytes = l.dz + align_up(BH * kD * 4);
  return l;
}

LinearBwdLayout linear_bwd_layout(int B, int nh, int64_t N) {
  return bwd_layout_of(linear_plan(B, nh, N), (size_t)B * nh);
}

cudaError_t launch_linear_bwd(const void* q, const void* k, const void* v, const void* dout, const void* saved,
                              void* dq, void* dk, void* dv, void* ws, int B, int nh, int64_t N, cudaStream_t st) {
  const LinearPlan p = linear_plan(B, nh, N);
  const int BH = B * nh;
  const LinearLayout fl = layout_of(p, BH);
  const LinearBwdLayout bl = bwd_layout_of(p, BH);
  const char* sv = static_cast<const char*>(saved);
  char* w = static_cast<char*>(ws);
  BQArgs qa;
  qa.N = (int)N;
  qa.BH = BH;
  qa.ntiles = p.ntiles;
  qa.chunk_tiles = p.b_chunk_tiles;
  qa.sum_tiles = p.sum_tiles;
  qa.sth = reinterpret_cast<const __nv_bfloat16*>(sv + fl.sth);
  qa.stl = reinterpret_cast<const __nv_bfloat16*>(sv + fl.stl);
  qa.zt = reinterpret_cast<const float*>(sv + fl.z);
  qa.part_dS = reinterpret_cast<float*>(w + bl.part_dS);
  qa.part_dz = reinterpret_cast<float*>(w + bl.part_dz);
  BCombArgs ca;
  ca.BH = BH;
  ca.chunks = p.b_chunks;
  ca.part_dS = qa.part_dS;
  ca.part_dz = qa.part_dz;
  ca.dsh = reinterpret_cast<__nv_bfloat16*>(w + bl.dsh);
  ca.dsl = reinterpret_cast<__nv_bfloat16*>(w + bl.dsl);
  ca.dsth = reinterpret_cast<__nv_bfloat16*>(w + bl.dsth);
  ca.dstl = reinterpret_cast<__nv_bfloat16*>(w + bl.dstl);
  ca.dz = reinterpret_cast<float*>(w + bl.dz);
  BKArgs ka;
  ka.ntiles = p.ntiles;
  ka.tiles_per_cta = p.b_chunk_tiles;
  ka.dsh = ca.dsh;
  ka.dsl = ca.dsl;
  ka.dsth = ca.dsth;
  ka.dstl = ca.dstl;
  ka.dz = ca.dz;

  CUtensorMap mq, mg, mk, mv, mdq, mdk, mdv;
  if (!make_tmap_5d(&mq, q, kD, (int)N, 1, 1, BH, kTile, 1, 1) || !make_tmap_5d(&mg, dout, kD, (int)N, 1, 1, BH, kTile, 1, 1) ||
      !make_tmap_5d(&mk, k, kD, (int)N, 1, 1, BH, kTile, 1, 1) || !make_tmap_5d(&mv, v, kD, (int)N, 1, 1, BH, kTile, 1, 1) ||
      !make_tmap_5d(&mdq, dq, kD, (int)N, 1, 1, BH, 32, 1, 1, 32) || !make_tmap_5d(&mdk, dk, kD, (int)N, 1, 1, BH, 32, 1, 1) ||
      !make_tmap_5d(&mdv, dv, kD, (int)N, 1, 1, BH, 32, 1, 1))
    return cudaErrorInvalidValue;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(la_bwd_query_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBQSmem)) !=
          cudaSuccess ||
      (e = cudaFuncSetAttribute(la_bwd_key_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBKSmem)) !=
          cudaSuccess)
    return e;
  prof_begin(kKLinearBwdQuery, st);
  la_bwd_query_kernel<<<dim3(p.b_chunks, BH), kThreadsB, kBQSmem, st>>>(mq, mg, mdq, qa);
  e = cudaGetLastError();
  prof_end(kKLinearBwdQuery, st);
  if (e != cudaSuccess) return e;
  prof_begin(kKLinearBwdCombine, st);
  la_bwd_combine_kernel<<<dim3(BH, (kD * kD + kD + 255) / 256), 256, 0, st>>>(ca);
  e = cudaGetLastError();
  prof_end(kKLinearBwdCombine, st);
  if (e != cudaSuccess) return e;
  prof_begin(kKLinearBwdKey, st);
  la_bwd_key_kernel<<<dim3(p.b_chunks, BH), kThreadsB, kBKSmem, st>>>(
      mk, mv, mdk, mdv, ka);
  e = cudaGetLastError();
  prof_end(kKLinearBwdKey, st);
  return e;
}

}  // namespace gattn
