// sm103_bwd_common.cuh -- pieces shared by the tensor-core backward kernels
// (sm103_bwd64.cu: d = 64; sm103_bwd.cu: d = 128).  Each including translation unit gets its own
// copy (anonymous namespace) and defines its own status word and WAIT().
#pragma once
#include "internal.cuh"
#include "sm103_common.cuh"

namespace gattn {
namespace {
using namespace sm103;

struct BwdArgs {
  Geom g;
  const float* lse2c;
  const float* dd;
  const int32_t* dst;  // per slot: token of a single-cover row, -2 multiply covered, -1 outside the tile
  const int32_t* nbt;  // boxes per tile
  const uint4* ext;  // dK/dV kernels: per-slot B-operand rows of the statistics (see bwd_prep)
  void* dq;
  void* dk;
  void* dv;
  float* dq_s;
  float* dk_s;
  float* dv_s;
  int items;  // B*nh * ntiles * nbmax_tot
};

__device__ __forceinline__ void decode_item(const Geom& g, int w, int& bh, int& tile, int& blk) {
  const int r = fdiv(w, g.fnb);
  blk = w - r * g.nbmax_tot;
  bh = fdiv(r, g.fntiles);
  tile = r - bh * g.ntiles;
}

// The first item at or after w whose box exists: the tile's boxes, 0 if there is
// none.  The math warps take this and the rows' places (dst) from what the prep
// pass wrote: 16 warps each working them out cost an item about 500 cycles (24 x
// 24 tiles, 16 heads: dK/dV kernel 3.01 -> 2.94 ms, dQ 2.40 -> 2.23).
__device__ __forceinline__ int next_boxes(const BwdArgs& a, int& w) {
  for (; w < a.items; w += gridDim.x) {
    int bh, tile, blk;
    decode_item(a.g, w, bh, tile, blk);
    const int nb = a.nbt[tile];
    if (blk < nb) return nb;
  }
  return 0;
}
// batch*head of item w
__device__ __forceinline__ int item_bh(const Geom& g, int w) { return fdiv(fdiv(w, g.fnb), g.fntiles); }

// byte offset of K-step ks (16 elements) in a 128-byte-swizzled K-major operand
__device__ __forceinline__ uint32_t kmaj_off(int ks) { return (ks >> 2) * 16384 + (ks & 3) * 32; }

// Warp roles of both backward kernels: warp 0 TMA producer, warp 1 TMEM
// allocator + issuer of the score products, warp kIssuerA issuer of the
// gradient products, warps kMath0.. elementwise math + epilogue (four per TMEM
// lane quadrant, each taking 32 of a row's 128 score columns).
constexpr int kMathW = 16;
constexpr int kMath0 = 3;
constexpr int kIssuerA = 2;
constexpr int kThreadsB = 32 * (kMath0 + kMathW);

// N FP32 columns of this thread's row, already in registers and scaled, to the
// output row (16 bytes at a time)
template <int N>
__device__ __forceinline__ void store_cols(float* out, const uint32_t (&r)[N]) {
#pragma unroll
  for (int e = 0; e < N; e += 4) *reinterpret_cast<uint4*>(out + e) = make_uint4(r[e], r[e + 1], r[e + 2], r[e + 3]);
}
template <int N>
__device__ __forceinline__ void store_cols(__nv_bfloat16* out, const uint32_t (&r)[N]) {
#pragma unroll
  for (int e = 0; e < N; e += 8)
    *reinterpret_cast<uint4*>(out + e) =
        make_uint4(pack_bf16(__uint_as_float(r[e]), __uint_as_float(r[e + 1])),
                   pack_bf16(__uint_as_float(r[e + 2]), __uint_as_float(r[e + 3])),
                   pack_bf16(__uint_as_float(r[e + 4]), __uint_as_float(r[e + 5])),
                   pack_bf16(__uint_as_float(r[e + 6]), __uint_as_float(r[e + 7])));
}

// Multiplies N accumulator columns by `mul` and writes them out: to `out` if
// this thread's row is covered by one tile only, and (the warp's 32 rows
// together, as soon as one of them is multiply covered) to the FP32 slots,
// through the warp's staging block `st` in shared memory and one TMA store of
// 32 rows x N columns at (row srow, column col).  A thread per row storing
// its own slot row touches 32 lines per instruction; the staged form writes
// whole 64- or 128-byte segments and leaves the waiting to the copy unit (16
// heads of 1024 tiles of 24 x 24 tokens: dK/dV kernel 3.96 -> 3.17 ms, dQ
// 3.35 -> 3.13).
// Rows at or past R are not staged (the block may be padding of an operand
// that has to stay zero), and slots of rows that are not multiply covered are
// never read.  Returns after issuing; lane 0 owns the bulk group.
template <int N, typename OutT>
__device__ __forceinline__ void row_out(uint32_t (&r)[N], float mul, bool valid, bool single, bool stage, OutT* out,
                                        const CUtensorMap* map, uint32_t st, int lane, int col, int srow) {
  static_assert(N == 16 || N == 32, "a staged row is 64 or 128 bytes");
#pragma unroll
  for (int e = 0; e < N; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * mul);
  if (single) store_cols<N>(out, r);
  if (!__any_sync(0xffffffffu, valid && !single)) return;
  if (stage) {
#pragma unroll
    for (int c = 0; c < N / 4; ++c) {
      const int sc = N == 32 ? c ^ (lane & 7) : c ^ ((lane >> 1) & 3);  // 128- or 64-byte swizzle
      st_shared_v4(st + lane * N * 4 + (sc << 4), r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
    }
  }
  fence_proxy_async_smem();
  __syncwarp();
  if (lane == 0) {
    tma_store_2d(map, st, col, srow);
    bulk_commit();
  }
}

// Multiplies 32 accumulator columns by `mul` and writes them out, to `out` if
// this thread's row is covered by one tile only, and (the warp's 32 rows
// together, as soon as one of them is multiply covered) to the FP32 slots from
// row 0 of the warp at `scr`; slots of other rows are never read.  The d = 128
// kernels have no shared memory for staged stores (row_out above); the
// transposed stores take a quarter of the LSU time of a thread writing its
// own row.
template <typename OutT>
__device__ __forceinline__ void row_slots(uint32_t (&r)[32], float mul, bool valid, bool single, OutT* out, float* scr,
                                          int lane) {
#pragma unroll
  for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * mul);
  if (single) store_cols<32>(out, r);
  if (!__any_sync(0xffffffffu, valid && !single)) return;
  store_rows16(scr, 128, lane, r);
  store_rows16(scr + 16, 128, lane, r + 16);
}

// dK/dV: P'^T of 32 columns of this thread's key row (S'^T already carries the
// statistics): FP32 in place of the scores, and as BF16 pairs.
__device__ __forceinline__ void kv_p(uint32_t (&s)[32], uint64_t s2, uint32_t (&pp)[16]) {
#pragma unroll
  for (int c = 0; c < 32; c += 2) {
    float a0, a1;
    f2unpack(fmul2(u2pack(s[c], s[c + 1]), s2), a0, a1);
    const float p0 = ex2(a0), p1 = ex2(a1);
    s[c] = __float_as_uint(p0);
    s[c + 1] = __float_as_uint(p1);
    pp[c >> 1] = pack_bf16(p0, p1);
  }
}
// dK/dV: dS^T = P'^T dP'^T (dP'^T already carries -D) as BF16 pairs
__device__ __forceinline__ void kv_ds(const uint32_t (&p)[32], const uint32_t (&dp)[32], uint32_t (&pd)[16]) {
#pragma unroll
  for (int c = 0; c < 32; c += 2) {
    float e0, e1;
    f2unpack(fmul2(u2pack(p[c], p[c + 1]), u2pack(dp[c], dp[c + 1])), e0, e1);
    pd[c >> 1] = pack_bf16(e0, e1);
  }
}

// dQ: P' = exp2(s S log2e - lse') of 32 columns of this thread's query row,
// FP32 in place of the scores
__device__ __forceinline__ void q_p(uint32_t (&s)[32], float sl2, float nL) {
  const uint64_t s2 = f2pack(sl2, sl2), nl2 = f2pack(nL, nL);
#pragma unroll
  for (int c = 0; c < 32; c += 2) {
    float a0, a1;
    f2unpack(ffma2(u2pack(s[c], s[c + 1]), s2, nl2), a0, a1);
    s[c] = __float_as_uint(ex2(a0));
    s[c + 1] = __float_as_uint(ex2(a1));
  }
}
// dQ: dS = P' (dP - D) as BF16 pairs
__device__ __forceinline__ void q_ds(const uint32_t (&p)[32], const uint32_t (&dp)[32], float nD, uint32_t (&pk)[16]) {
  const uint64_t nd2 = f2pack(nD, nD);
#pragma unroll
  for (int c = 0; c < 32; c += 2) {
    float e0, e1;
    f2unpack(fmul2(u2pack(p[c], p[c + 1]), fadd2(u2pack(dp[c], dp[c + 1]), nd2)), e0, e1);
    pk[c >> 1] = pack_bf16(e0, e1);
  }
}

// Constant A operands of the extension steps, K-major without swizzle: 128
// rows x 16 B (K-columns 0..7) followed by 2 KB of zeros (K-columns 8..15).
// `n` blocks of 4 KB from `base`: block 0 has ones in K 0..2 (dK/dV: adds x of
// the statistics row) or in K 0 (dQ: adds the key bias), block 1 ones in K
// 3..5 (dK/dV: adds y).  Then `nz` further 4 KB B-operand blocks at `zb`
// whose zero halves are cleared (their first 2 KB is loaded per box).
__device__ __forceinline__ void init_ext_operands(uint8_t* base, int n, bool stats, uint8_t* zb, int nz) {
  for (int r = threadIdx.x; r < n * 256 + nz * 128; r += blockDim.x) {
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    uint8_t* dst;
    if (r < n * 256) {
      const int blk = r >> 8, rr = r & 255;
      if (rr < 128) {
        if (!stats)
          v = make_uint4(0x00003F80u, 0u, 0u, 0u);                                      // (1, 0, ..., 0)
        else
          v = blk == 0 ? make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u)                   // (1, 1, 1, 0, 0, 0, 0, 0)
                       : make_uint4(0u, 0x3F800000u, 0x3F803F80u, 0u);                  // (0, 0, 0, 1, 1, 1, 0, 0)
      }
      dst = base + blk * 4096 + rr * 16;
    } else {
      const int q = r - n * 256;
      dst = zb + (q >> 7) * 4096 + 2048 + (q & 127) * 16;
    }
    *reinterpret_cast<uint4*>(dst) = v;
  }
}

}  // namespace
}  // namespace gattn
