// simt_fp32.cu -- the plain FP32 form of STORM-GPA tile attention (CUDA cores,
// no tensor cores): forward (online softmax, Sec. III-C / III-D Level 5) and
// the two backward kernels (dQ per query row, dK/dV per key row).  This is
// the FP32 baseline the BF16 tensor-core form is measured against, and the
// path used when the inputs are FP32.
//
// Work decomposition: one CTA per (row block, tile, batch*head); a warp owns
// 8 RG rows of the extended tile, keys (or queries, for dK/dV) stream through
// shared memory 64 at a time (32 for short tiles, see with_shape).  Both kinds of products are register-tiled, 8
// rows per thread, and issue packed FP32 pairs (fma.rn.f32x2), so that the FMA
// pipe is the limit and not the issue slots or the shared-memory reads:
//   scores   8 rows x KT keys a thread, contraction over d in pairs of
//            neighbouring elements (both operands are d-contiguous, so pairs
//            load as they lie; the two partial sums are added at the end);
//            12 16-byte loads per 64 pair instructions at d = 64
//   P V, ... 8 rows x CT columns a thread in pairs of rows, one key at a time;
//            the warp's P is kept key-major, so a key's rows load as pairs, and
//            the CT values of the other operand are doubled in registers; 3
//            loads per 16 pair instructions (with P doubled in shared memory
//            instead, 5: the loads, not the FMAs, then set the pace)
// Rows never leave their warp: P goes through a warp-private buffer, so CTA
// barriers only order the streamed blocks.  Every streamed block is reduced
// locally before it is folded into the running sums (two-level summation,
// which keeps the FP32 error of L-long sums near eps * (sqrt(64) + sqrt(L/64))).
// Bound: the FP32 pipe (128 lanes a clock and SM), 53-57 % active with two
// warps per scheduler (registers), shared memory at half its rate.  4 heads of
// a 4 x 64 x 128 clip in 16 tiles of up to 4608 tokens, d = 64: forward 14.6 ->
// 6.2 ms, dQ 17.0 -> 8.8, dK/dV 19.4 -> 10.9 (before: a thread group per row,
// one FMA per shared-memory word).
#include "internal.cuh"
#include "sm103_common.cuh"

GATTN_DEFINE_STATUS(simt)

namespace gattn {
namespace {
using sm103::f2pack;
using sm103::f2unpack;
using sm103::fadd2;
using sm103::ffma2;
using sm103::fmul2;

// Shape of the kernels at head size D with W warps per CTA, RG row groups of 8
// rows per warp and BN streamed rows per block.
template <int D_, int W_, int RG_, int BN_ = 64>
struct Shape {
  static constexpr int D = D_, W = W_, RG = RG_, BN = BN_;
  static constexpr int LG = 32 / RG;            // lanes of a row group
  static constexpr int KT = BN / LG;            // score columns per thread: keys lg + LG * jj
  static constexpr int CT = D / LG;             // output columns per thread: CT * lg ...
  static constexpr int WR = 8 * RG;             // rows per warp
  static constexpr int BM = W * WR;             // rows per CTA
  static constexpr int T = 32 * W;
  static constexpr int LD = D + 4;              // padded row of a staged matrix (floats): conflict-free column walks
  static constexpr int HJ = KT == 1 || (RG == 1 && D == 64) ? 1 : 2;  // score columns per thread exchanged at a time
  static constexpr int HK = HJ * LG;            // keys of P exchanged at a time
  static constexpr int NH = BN / HK;
  // resident CTAs per SM (registers, shared memory)
  static constexpr int CTAS = D == 128 ? (BN == 64 ? 1 : W == 2 ? 3 : 2) : D == 64 ? (BN == 64 ? 2 : 4) : BN == 32 ? 16 / W : W == 4 ? 3 : 2;
  static constexpr bool SKIP = BN < 64;         // warps without a row of the tile only stage
  static constexpr int PB = WR + 4;             // floats per key of the P buffer, padded
  static constexpr int PW = HK * PB;            // floats of a warp's P buffer
};

// Tile-row tokens: row r of the extended tile by FP32 quotients (box_index).
__device__ __forceinline__ int64_t row_token(const Geom& g, const TileBox& tb, int r, int l[3]) {
  box_index(r, tb.e[1], tb.e[2], l[0], l[1], l[2]);
  return grid_token(g, tb, l);
}

__device__ __forceinline__ void cp16(float* dst, const float* src, bool ok) {
  const int n = ok ? 16 : 0;  // 0: the 16 bytes are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sm103::smem_u32(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Rows [j0, j0 + ROWS) of the tile of a [N, D] tensor into padded rows (zeros past the tile).
template <class S, int ROWS>
__device__ __forceinline__ void stage(const Geom& g, const TileBox& tb, int j0, const float* __restrict__ A, float* As) {
  constexpr int F4 = S::D / 4;
#pragma unroll 4
  for (int idx = threadIdx.x; idx < ROWS * F4; idx += S::T) {
    const int jj = idx / F4, f = idx % F4;
    const bool ok = j0 + jj < tb.L;
    int l[3];
    const int64_t tok = row_token(g, tb, ok ? j0 + jj : 0, l);
    cp16(As + jj * S::LD + 4 * f, A + tok * S::D + 4 * f, ok);
  }
}

// acc[i][jj] = rows[i] . cols[lg + LG jj]: 8 rows from `rows` (this thread's row
// group), KT columns.
template <class S>
__device__ __forceinline__ void dots(const float* __restrict__ rows, const float* __restrict__ cols, int lg,
                                     float (&s)[8][S::KT]) {
  uint64_t acc[8][S::KT];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < S::KT; ++j) acc[i][j] = 0;
  const float* cp = cols + lg * S::LD;
#pragma unroll 2
  for (int k = 0; k < S::D; k += 4) {
    ulonglong2 b[S::KT];
#pragma unroll
    for (int j = 0; j < S::KT; ++j) b[j] = *reinterpret_cast<const ulonglong2*>(cp + j * S::LG * S::LD + k);
    // four rows at a time: an accumulator's two updates are 4 KT instructions apart
#pragma unroll
    for (int i0 = 0; i0 < 8; i0 += 4) {
      ulonglong2 a[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const ulonglong2*>(rows + (i0 + i) * S::LD + k);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < S::KT; ++j) acc[i0 + i][j] = ffma2(a[i].x, b[j].x, acc[i0 + i][j]);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < S::KT; ++j) acc[i0 + i][j] = ffma2(a[i].y, b[j].y, acc[i0 + i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < S::KT; ++j) {
      float x, y;
      f2unpack(acc[i][j], x, y);
      s[i][j] = x + y;
    }
}

// Accumulators of 8 rows x CT columns: pairs of rows (2 i, 2 i + 1).
template <class S>
using Acc = uint64_t[4][S::CT];

// out[i][c] += sum over the block's 64 keys of p[row][key] * M[key][CT lg + c],
// p being this thread's score columns (exchanged within the warp through pb).
template <class S>
__device__ __forceinline__ void axpys(const float (&p)[8][S::KT], const float* __restrict__ M, float* pb, int rg, int lg,
                                      Acc<S>& out) {
  Acc<S> acc;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < S::CT; ++c) acc[i][c] = 0;
#pragma unroll
  for (int h = 0; h < S::NH; ++h) {
    __syncwarp();  // the previous half (or product) has been read
#pragma unroll
    for (int jj = 0; jj < S::HJ; ++jj) {
      float4* d = reinterpret_cast<float4*>(pb + (lg + S::LG * jj) * S::PB + 8 * rg);
      const int j = S::HJ * h + jj;
      d[0] = make_float4(p[0][j], p[1][j], p[2][j], p[3][j]);
      d[1] = make_float4(p[4][j], p[5][j], p[6][j], p[7][j]);
    }
    __syncwarp();
    const float* m = M + h * S::HK * S::LD + S::CT * lg;
    const float* pp = pb + 8 * rg;
#pragma unroll 4
    for (int key = 0; key < S::HK; ++key) {
      uint64_t v[S::CT];
      if constexpr (S::CT == 4) {
        const float4 t = *reinterpret_cast<const float4*>(m + key * S::LD);
        v[0] = f2pack(t.x, t.x);
        v[1] = f2pack(t.y, t.y);
        v[2] = f2pack(t.z, t.z);
        v[3] = f2pack(t.w, t.w);
      } else {
        const float2 t = *reinterpret_cast<const float2*>(m + key * S::LD);
        v[0] = f2pack(t.x, t.x);
        v[1] = f2pack(t.y, t.y);
      }
      const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(pp + key * S::PB);
      const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(pp + key * S::PB + 4);
#pragma unroll
      for (int c = 0; c < S::CT; ++c) {
        acc[0][c] = ffma2(a.x, v[c], acc[0][c]);
        acc[1][c] = ffma2(a.y, v[c], acc[1][c]);
        acc[2][c] = ffma2(b.x, v[c], acc[2][c]);
        acc[3][c] = ffma2(b.y, v[c], acc[3][c]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < S::CT; ++c) out[i][c] = fadd2(out[i][c], acc[i][c]);
}

template <class S>
__device__ __forceinline__ void zero_acc(Acc<S>& a) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < S::CT; ++c) a[i][c] = 0;
}

// the CT accumulated columns of row i, times mul, to the output row or the slot row
template <class S, typename T>
__device__ __forceinline__ void store_cols(T* dst, const Acc<S>& a, int i, float mul) {
  float x[S::CT];
#pragma unroll
  for (int c = 0; c < S::CT; ++c) {
    float u, v;
    f2unpack(a[i >> 1][c], u, v);
    x[c] = i & 1 ? v : u;
  }
  if constexpr (S::CT == 4) {
    store4<T>(dst, make_float4(x[0] * mul, x[1] * mul, x[2] * mul, x[3] * mul));
  } else if constexpr (sizeof(T) == 2) {
    *reinterpret_cast<__nv_bfloat162*>(dst) = __floats2bfloat162_rn(x[0] * mul, x[1] * mul);
  } else {
    *reinterpret_cast<float2*>(dst) = make_float2(x[0] * mul, x[1] * mul);
  }
}

template <int LG>
__device__ __forceinline__ float group_max(float v) {
#pragma unroll
  for (int o = 1; o < LG; o <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
template <int LG>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int o = 1; o < LG; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------- forward
template <class S>
struct FwdSmem {
  float q[S::BM * S::LD];
  float k[2][S::BN * S::LD];
  float v[2][S::BN * S::LD];
  float p[S::W][S::PW];
};

template <class S, typename OutT>
__global__ void __launch_bounds__(S::T, S::CTAS) simt_fwd_kernel(const Geom g, const float* __restrict__ Q,
                                                        const float* __restrict__ K, const float* __restrict__ V,
                                                        OutT* __restrict__ out, float* __restrict__ lse2,
                                                        float* __restrict__ ot) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  auto& sm = *reinterpret_cast<FwdSmem<S>*>(smem_raw);
  const int tile = blockIdx.y, bh = blockIdx.z;
  TileBox tb;
  tile_box(g, tile, tb);
  const int row0 = blockIdx.x * S::BM;
  if (row0 >= tb.L) return;  // uniform over the CTA
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rg = lane / S::LG, lg = lane % S::LG;
  const int64_t base = (int64_t)bh * g.N * S::D;
  stage<S, S::BM>(g, tb, row0, Q + base, sm.q);
  stage<S, S::BN>(g, tb, 0, K + base, sm.k[0]);
  stage<S, S::BN>(g, tb, 0, V + base, sm.v[0]);
  cp_commit();
  const bool busy = row0 + warp * S::WR < tb.L;  // the warp has a row of the tile
  const int r0 = warp * S::WR + rg * 8;  // first of this thread's 8 rows within the CTA
  float* pb = sm.p[warp];

  Acc<S> o;
  zero_acc<S>(o);
  float m[8], l[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
  }
  for (int j0 = 0, b = 0; j0 < tb.L; j0 += S::BN, b ^= 1) {
    cp_wait<0>();
    __syncthreads();  // block j0 is staged, block j0 - 64 has been read by every warp
    if (j0 + S::BN < tb.L) {
      stage<S, S::BN>(g, tb, j0 + S::BN, K + base, sm.k[b ^ 1]);
      stage<S, S::BN>(g, tb, j0 + S::BN, V + base, sm.v[b ^ 1]);
      cp_commit();
    }
    if (S::SKIP && !busy) continue;
    float s[8][S::KT];
    dots<S>(sm.q + r0 * S::LD, sm.k[b], lg, s);
#pragma unroll
    for (int j = 0; j < S::KT; ++j) {
      const bool in = j0 + lg + S::LG * j < tb.L;
#pragma unroll
      for (int i = 0; i < 8; ++i) s[i][j] = in ? s[i][j] * g.scale_log2 : -INFINITY;
    }
    float alpha[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float mx = s[i][0];
#pragma unroll
      for (int j = 1; j < S::KT; ++j) mx = fmaxf(mx, s[i][j]);
      mx = fmaxf(m[i], group_max<S::LG>(mx));
      alpha[i] = exp2f(m[i] - mx);  // 0 on the first block (m = -inf)
      m[i] = mx;
      float lc = 0.f;
#pragma unroll
      for (int j = 0; j < S::KT; ++j) {
        s[i][j] = exp2f(s[i][j] - mx);
        lc += s[i][j];
      }
      l[i] = l[i] * alpha[i] + lc;  // this thread's keys; the group's sums are added at the end
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < S::CT; ++c) o[i][c] = fmul2(o[i][c], f2pack(alpha[2 * i], alpha[2 * i + 1]));
    axpys<S>(s, sm.v[b], pb, rg, lg, o);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float ls = group_sum<S::LG>(l[i]);
    const int r = row0 + r0 + i;
    if (r >= tb.L) continue;
    int lr[3];
    const int64_t tok = row_token(g, tb, r, lr);
    const int p[3] = {tb.lo[0] + lr[0], tb.lo[1] + lr[1], tb.lo[2] + lr[2]};
    const int64_t slot = slot_of(g, bh, tile, tb.e, lr);
    if (lg == 0) lse2[slot] = m[i] + log2f(ls);
    const float inv = 1.f / ls;
    if (only_cover(g, tb, p)) store_cols<S>(out + base + tok * S::D + S::CT * lg, o, i, inv);
    else store_cols<S>(ot + slot * S::D + S::CT * lg, o, i, inv);
  }
}

// ---------------------------------------------------------------- backward: dQ
// P = exp2(s q.k log2e - lse') already carries the merge weight w_t / sum w,
// so dS = P (dOut.v - D) and dQ_t = s sum_j dS k_j (the workspace holds -lse'
// and -D).  V of the next block is loaded while this block's dQ product runs,
// K one block ahead.
template <class S>
struct DqSmem {
  float q[S::BM * S::LD];
  float go[S::BM * S::LD];
  float k[2][S::BN * S::LD];
  float v[S::BN * S::LD];
  float p[S::W][S::PW];
};

template <class S, typename OutT>
__global__ void __launch_bounds__(S::T, S::CTAS) simt_dq_kernel(const Geom g, const float* __restrict__ Q,
                                                       const float* __restrict__ K, const float* __restrict__ V,
                                                       const float* __restrict__ dO, const float* __restrict__ lse2c,
                                                       const float* __restrict__ dd, OutT* __restrict__ dq,
                                                       float* __restrict__ dq_s) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  auto& sm = *reinterpret_cast<DqSmem<S>*>(smem_raw);
  const int tile = blockIdx.y, bh = blockIdx.z;
  TileBox tb;
  tile_box(g, tile, tb);
  const int row0 = blockIdx.x * S::BM;
  if (row0 >= tb.L) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rg = lane / S::LG, lg = lane % S::LG;
  const int64_t base = (int64_t)bh * g.N * S::D;
  stage<S, S::BM>(g, tb, row0, Q + base, sm.q);
  stage<S, S::BM>(g, tb, row0, dO + base, sm.go);
  stage<S, S::BN>(g, tb, 0, K + base, sm.k[0]);
  stage<S, S::BN>(g, tb, 0, V + base, sm.v);
  cp_commit();
  const bool busy = row0 + warp * S::WR < tb.L;  // the warp has a row of the tile
  const int r0 = warp * S::WR + rg * 8;
  float nL[8], nD[8];  // -lse' and -D (negated in the workspace)
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = row0 + r0 + i;
    nL[i] = -INFINITY;
    nD[i] = 0.f;
    if (r < tb.L) {
      int lr[3];
      row_token(g, tb, r, lr);
      const int64_t slot = slot_of(g, bh, tile, tb.e, lr);
      nL[i] = lse2c[slot];
      nD[i] = dd[slot];
    }
  }
  Acc<S> acc;
  zero_acc<S>(acc);
  for (int j0 = 0, b = 0; j0 < tb.L; j0 += S::BN, b ^= 1) {
    const bool more = j0 + S::BN < tb.L;
    cp_wait<0>();
    __syncthreads();  // block j0 is staged, the other K buffer has been read
    if (more) stage<S, S::BN>(g, tb, j0 + S::BN, K + base, sm.k[b ^ 1]);
    float s[8][S::KT], dp[8][S::KT];
    if (!S::SKIP || busy) {
      dots<S>(sm.q + r0 * S::LD, sm.k[b], lg, s);
#pragma unroll
      for (int j = 0; j < S::KT; ++j) {
        const bool in = j0 + lg + S::LG * j < tb.L;
#pragma unroll
        for (int i = 0; i < 8; ++i) s[i][j] = in ? exp2f(fmaf(s[i][j], g.scale_log2, nL[i])) : 0.f;
      }
      dots<S>(sm.go + r0 * S::LD, sm.v, lg, dp);
    }
    __syncthreads();  // V has been read
    if (more) {
      stage<S, S::BN>(g, tb, j0 + S::BN, V + base, sm.v);
      cp_commit();
    }
    if (S::SKIP && !busy) continue;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < S::KT; ++j) s[i][j] *= dp[i][j] + nD[i];
    axpys<S>(s, sm.k[b], sm.p[warp], rg, lg, acc);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = row0 + r0 + i;
    if (r >= tb.L) continue;
    int lr[3];
    const int64_t tok = row_token(g, tb, r, lr);
    const int p[3] = {tb.lo[0] + lr[0], tb.lo[1] + lr[1], tb.lo[2] + lr[2]};
    if (only_cover(g, tb, p)) store_cols<S>(dq + base + tok * S::D + S::CT * lg, acc, i, g.scale);
    else store_cols<S>(dq_s + slot_of(g, bh, tile, tb.e, lr) * S::D + S::CT * lg, acc, i, g.scale);
  }
}

// ---------------------------------------------------------------- backward: dK, dV
// Rows are keys: dV_t(j) = sum_i P_ij dOut_i, dK_t(j) = s sum_i dS_ij q_i.
// dOut of the next block is loaded while this block's dK product runs, Q one
// block ahead.
template <class S>
struct DkvSmem {
  float k[S::BM * S::LD];
  float v[S::BM * S::LD];
  float q[2][S::BN * S::LD];
  float go[S::BN * S::LD];
  float p[S::W][S::PW];
  float nL[2][S::BN], nD[2][S::BN];
};

template <class S, typename OutT>
__global__ void __launch_bounds__(S::T, S::CTAS) simt_dkdv_kernel(const Geom g, const float* __restrict__ Q,
                                                         const float* __restrict__ K, const float* __restrict__ V,
                                                         const float* __restrict__ dO, const float* __restrict__ lse2c,
                                                         const float* __restrict__ dd, OutT* __restrict__ dk,
                                                         OutT* __restrict__ dv, float* __restrict__ dk_s,
                                                         float* __restrict__ dv_s) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  auto& sm = *reinterpret_cast<DkvSmem<S>*>(smem_raw);
  const int tile = blockIdx.y, bh = blockIdx.z;
  TileBox tb;
  tile_box(g, tile, tb);
  const int row0 = blockIdx.x * S::BM;
  if (row0 >= tb.L) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rg = lane / S::LG, lg = lane % S::LG;
  const int64_t base = (int64_t)bh * g.N * S::D;
  // -lse' and -D of the block's queries; rows past the tile get P = 0
  auto stats = [&](int i0, int b) {
    for (int t = threadIdx.x; t < S::BN; t += S::T) {
      float a = -INFINITY, d = 0.f;
      if (i0 + t < tb.L) {
        int lr[3];
        row_token(g, tb, i0 + t, lr);
        const int64_t slot = slot_of(g, bh, tile, tb.e, lr);
        a = lse2c[slot];
        d = dd[slot];
      }
      sm.nL[b][t] = a;
      sm.nD[b][t] = d;
    }
  };
  stage<S, S::BM>(g, tb, row0, K + base, sm.k);
  stage<S, S::BM>(g, tb, row0, V + base, sm.v);
  stage<S, S::BN>(g, tb, 0, Q + base, sm.q[0]);
  stage<S, S::BN>(g, tb, 0, dO + base, sm.go);
  cp_commit();
  stats(0, 0);
  const bool busy = row0 + warp * S::WR < tb.L;  // the warp has a row of the tile
  const int r0 = warp * S::WR + rg * 8;
  Acc<S> adk, adv;
  zero_acc<S>(adk);
  zero_acc<S>(adv);
  for (int i0 = 0, b = 0; i0 < tb.L; i0 += S::BN, b ^= 1) {
    const bool more = i0 + S::BN < tb.L;
    cp_wait<0>();
    __syncthreads();  // block i0 is staged, the other Q buffer has been read
    if (more) {
      stage<S, S::BN>(g, tb, i0 + S::BN, Q + base, sm.q[b ^ 1]);
      stats(i0 + S::BN, b ^ 1);
    }
    float s[8][S::KT], dp[8][S::KT];
    if (!S::SKIP || busy) {
      dots<S>(sm.k + r0 * S::LD, sm.q[b], lg, s);
#pragma unroll
      for (int j = 0; j < S::KT; ++j) {
        const float nL = sm.nL[b][lg + S::LG * j];
#pragma unroll
        for (int i = 0; i < 8; ++i) s[i][j] = exp2f(fmaf(s[i][j], g.scale_log2, nL));
      }
      if (i0 + S::BN > tb.L) {
        // rows past the tile are zeros, which an infinite key turns into NaN: P = 0 whatever the key is
#pragma unroll
        for (int j = 0; j < S::KT; ++j)
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (i0 + lg + S::LG * j >= tb.L) s[i][j] = 0.f;
      }
      axpys<S>(s, sm.go, sm.p[warp], rg, lg, adv);
      dots<S>(sm.v + r0 * S::LD, sm.go, lg, dp);
    }
    __syncthreads();  // dOut has been read
    if (more) {
      stage<S, S::BN>(g, tb, i0 + S::BN, dO + base, sm.go);
      cp_commit();
    }
    if (S::SKIP && !busy) continue;
#pragma unroll
    for (int j = 0; j < S::KT; ++j) {
      const float nD = sm.nD[b][lg + S::LG * j];
#pragma unroll
      for (int i = 0; i < 8; ++i) s[i][j] *= dp[i][j] + nD;
    }
    axpys<S>(s, sm.q[b], sm.p[warp], rg, lg, adk);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = row0 + r0 + i;
    if (r >= tb.L) continue;
    int lr[3];
    const int64_t tok = row_token(g, tb, r, lr);
    const int p[3] = {tb.lo[0] + lr[0], tb.lo[1] + lr[1], tb.lo[2] + lr[2]};
    if (only_cover(g, tb, p)) {
      store_cols<S>(dk + base + tok * S::D + S::CT * lg, adk, i, g.scale);
      store_cols<S>(dv + base + tok * S::D + S::CT * lg, adv, i, 1.f);
    } else {
      const int64_t slot = slot_of(g, bh, tile, tb.e, lr);
      store_cols<S>(dk_s + slot * S::D + S::CT * lg, adk, i, g.scale);
      store_cols<S>(dv_s + slot * S::D + S::CT * lg, adv, i, 1.f);
    }
  }
}

template <typename Kern>
cudaError_t smem_limit(Kern k, size_t bytes) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <class S, typename OutT>
cudaError_t fwd_run(const Geom& g, const float* q, const float* k, const float* v, void* out, float* lse2, float* ot,
                    cudaStream_t st) {
  const dim3 grid((g.Lmax + S::BM - 1) / S::BM, g.ntiles, g.B * g.nh);
  auto kern = simt_fwd_kernel<S, OutT>;
  cudaError_t e = smem_limit(kern, sizeof(FwdSmem<S>));
  if (e != cudaSuccess) return e;
  kern<<<grid, S::T, sizeof(FwdSmem<S>), st>>>(g, q, k, v, static_cast<OutT*>(out), lse2, ot);
  return cudaGetLastError();
}

template <class S, typename OutT>
cudaError_t bwd_run(const Geom& g, const float* q, const float* k, const float* v, const float* dout,
                    const float* lse2c, const float* dd, void* dq, void* dk, void* dv, float* dq_s, float* dk_s,
                    float* dv_s, cudaStream_t st) {
  const dim3 grid((g.Lmax + S::BM - 1) / S::BM, g.ntiles, g.B * g.nh);
  auto k1 = simt_dq_kernel<S, OutT>;
  auto k2 = simt_dkdv_kernel<S, OutT>;
  cudaError_t e = smem_limit(k1, sizeof(DqSmem<S>));
  if (e == cudaSuccess) e = smem_limit(k2, sizeof(DkvSmem<S>));
  if (e != cudaSuccess) return e;
  prof_begin(kKBwdDq, st);
  k1<<<grid, S::T, sizeof(DqSmem<S>), st>>>(g, q, k, v, dout, lse2c, dd, static_cast<OutT*>(dq), dq_s);
  prof_end(kKBwdDq, st);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  prof_begin(kKBwdDkdv, st);
  k2<<<grid, S::T, sizeof(DkvSmem<S>), st>>>(g, q, k, v, dout, lse2c, dd, static_cast<OutT*>(dk),
                                             static_cast<OutT*>(dv), dk_s, dv_s);
  prof_end(kKBwdDkdv, st);
  return cudaGetLastError();
}

// Runs f with the shape for this problem.
//   Tiles of more than 32 rows: 64-row CTAs of warps with 16 rows (8 x 4 score
// tiles a thread: fewest shared-memory reads per FMA), or, where those would
// leave SMs without a CTA, 32-row CTAs of warps with 8 rows (8 x 2 tiles, twice
// the warps: a training step on one head of a 64 x 64 frame 285 us, 16-row warps
// 311; the 8-row form costs large problems 15 %).
//   Tiles of up to 32 rows: blocks of 32 rows and 32-row CTAs (16 rows at d = 128
// up to 16), twice as many of them per SM, whose warps without a row only stage.
// Blocks of 64 make such a tile pay for 64 x 64 scores: training steps of 4096
// tiles of 16 rows took 465, 660 and 1404 us at d = 32, 64 and 128, now 168, 252
// and 435; at 36 rows the larger blocks are ahead (d = 64 729 against 782).
//   d = 32: a product is too short to hide its loads with eight warps per SM, so
// blocks of 32 and four CTAs up to 448 rows (1024 tiles of 64 rows 154 -> 127 us,
// of 144 669 -> 536, 400-row tiles 802 -> 742), beyond them blocks of 64 and three.
template <int D, typename F>
cudaError_t with_shape(const Geom& g, F f) {
  const int64_t blocks = (int64_t)((g.Lmax + 63) / 64) * g.ntiles * g.B * g.nh;
  const bool many = blocks > num_sms();
  if constexpr (D == 128) {
    if (g.Lmax <= 16) return f(Shape<D, 2, 1, 32>());
    if (g.Lmax <= 32) return f(Shape<D, 4, 1, 32>());
    return many ? f(Shape<D, 8, 1>()) : f(Shape<D, 4, 1>());
  } else if constexpr (D == 64) {
    if (g.Lmax <= 32) return f(Shape<D, 4, 1, 32>());
    return many ? f(Shape<D, 4, 2>()) : f(Shape<D, 4, 1>());
  } else {
    if (g.Lmax <= 32) return f(Shape<D, 2, 2, 32>());
    if (!many) return f(Shape<D, 2, 2>());
    return g.Lmax <= 448 ? f(Shape<D, 4, 2, 32>()) : f(Shape<D, 4, 2>());
  }
}

template <typename F>
cudaError_t with_d(const Geom& g, F f) {
  switch (g.d) {
    case 32: return with_shape<32>(g, f);
    case 64: return with_shape<64>(g, f);
    case 128: return with_shape<128>(g, f);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_simt_fwd(const Geom& g, const float* q, const float* k, const float* v, void* out,
                            int out_dtype, float* lse2, float* ot, cudaStream_t st) {
  return with_d(g, [&](auto s) {
    using S = decltype(s);
    return out_dtype == GATTN_BF16 ? fwd_run<S, __nv_bfloat16>(g, q, k, v, out, lse2, ot, st)
                                   : fwd_run<S, float>(g, q, k, v, out, lse2, ot, st);
  });
}

cudaError_t launch_simt_bwd(const Geom& g, const float* q, const float* k, const float* v, const float* dout,
                            const float* lse2c, const float* dd, void* dq, void* dk, void* dv, int out_dtype,
                            float* dq_s, float* dk_s, float* dv_s, cudaStream_t st) {
  return with_d(g, [&](auto s) {
    using S = decltype(s);
    return out_dtype == GATTN_BF16
               ? bwd_run<S, __nv_bfloat16>(g, q, k, v, dout, lse2c, dd, dq, dk, dv, dq_s, dk_s, dv_s, st)
               : bwd_run<S, float>(g, q, k, v, dout, lse2c, dd, dq, dk, dv, dq_s, dk_s, dv_s, st);
  });
}

}  // namespace gattn
