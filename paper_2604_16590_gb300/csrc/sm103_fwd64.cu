// sm103_fwd64.cu -- BF16 tensor-core forward of STORM-GPA tile attention for
// head size d = 64 on GB300 (sm_103a): two query boxes per work item, each
// with its own scores, probabilities and output in tensor memory.
//
// Per extended tile t (arXiv 2604.16590, Sec. III-C) and pair of 128-query
// boxes (A, B) of the tile, the CTA streams the tile's 128-key boxes once for
// both query boxes (flash-style online softmax, the FlashAttention of
// Sec. III-D Level 5):
//   S_x  = Q_x K_j^T                    tcgen05, A = Q_x, B = K_j (both shared memory)
//   m_x  = max(m_x, rowmax(s S_x))      log2 domain, lazily moved (threshold 8)
//   P_x  = exp2(s S_x log2e - m_x)      BF16 pairs -> TMEM
//   O_x += P_x V_j                      tcgen05, A = P_x from TMEM, B = V_j (MN-major)
// A softmax thread reads its row's 128 scores into registers at once and
// releases S_x, so S_x(j+1) is computed while the exponentials of box j run;
// P_x(j) waits only for P V_x(j-1).  With two boxes in flight the tensor pipe
// and the exp unit are busy at the same time.  The epilogue writes O / l for
// rows covered by one tile straight to the output and parks multiply-covered
// rows (FP32) for the deterministic Hann merge, and stores the row log-sum-exp.
//
// Warp roles (384 threads = three warpgroups, one CTA per SM, persistent over
// work items (batch*head, tile, box pair)):
//   warp 0        TMA producer (lane 0: Q_A, Q_B once per item; K_j, V_j through
//                 a ring) and key-mask writer (all lanes: for a key block with
//                 padding rows or rows outside the tile, the bias row of its
//                 stage, see below)
//   warp 1        TMEM allocator + issuer of the S products
//   warps 2, 3    issuers of the P V products, one per box.  A thread's mbarrier
//                 waits stall until its own issued MMAs have drained, which the
//                 other threads' MMAs in the pipe prolong: with one issuer for
//                 both boxes, P_A(j) lay finished for up to half a block while
//                 that thread still waited out P V_B(j-1) (16 heads of 1024
//                 tiles of 24 x 24: 2.03 -> 1.88 ms; tiles of 36864 tokens, where
//                 the softmax threads' own chain sets the pace, 58.4 ms either way)
//   warps 4..7    softmax + epilogue of box A, warps 8..11 of box B: one warp
//                 per TMEM lane quadrant, one thread per query row owning all
//                 128 key columns (no cross-warp reduction)
// Registers: the first warpgroup gives up registers (setmaxnreg) so that the
// softmax threads hold a whole row of scores: 128 x 72 + 2 x 128 x 216 =
// 384 x 168, the launch's allocation.
// TMEM (512 columns): S_x at 128 x, P_x at 256 + 64 x, O_x at 384 + 64 x.
//
// Key masking without a masked softmax: a key block that contains padding rows
// or keys outside the tile gets one more K = 16 step in its S product, a
// column of ones times the block's bias row (0 or -1e30 per key), so the
// masked scores arrive as -1e30 and their probabilities are exactly 0.  The
// softmax threads then run one branch-free form for every block (a second,
// masked form of the exponential loop measured 19 % slower even where it was
// never taken).
//
// Ragged mode (the serving engine): the work items of all active requests in
// one launch; each item resolves through the request table in device memory
// (tensor map over the request's state z = Q = K = V, geometry, outputs), and
// the producer acquires a request's tensor map before its first load from it.
#include <string.h>

#include "internal.cuh"
#include "sm103_common.cuh"

GATTN_DEFINE_STATUS(sm103_fwd64)

namespace gattn {
namespace {
using namespace sm103;

__device__ void set_status_f64(uint32_t c) { set_status(c); }
#define WAIT(bar, par) mbar_wait<set_status_f64>((bar), (par), abort_flag)

constexpr int kD = 64;
constexpr int kBox = 128 * kD * 2;  // one 128-token box of one operand, BF16, 16 KB
constexpr int kSoft0 = 4;           // first softmax warp
constexpr int kThreadsF = 384;
constexpr uint32_t kRegsLow = 72, kRegsHigh = 216;  // 128 x 72 + 256 x 216 = 384 x 168
constexpr float kRescaleLog2 = 8.f;

template <bool RAGGED>
struct Cfg {
  static constexpr int kStages = RAGGED ? 4 : 3;  // K/V ring depth: the staged outputs take a stage
  // two Q buffers (items alternate): buffer b holds Q_A at kQ + 2 b kBox, Q_B after it
  static constexpr int kQ = 0;
  static constexpr int kK = 4 * kBox;
  static constexpr int kV = kK + kStages * kBox;
  // Key-mask extension operands, K-major without swizzle (128 rows x 16 B,
  // then 2 KB of zeros for K-columns 8..15): the A operand has 1 in K-column 0
  // of every row; stage s of the B operand holds the key block's bias
  // (0 for a key of the tile, -1e30 for a padding row or a key outside it).
  static constexpr int kOut = kV + kStages * kBox;  // staged output columns 32..63, 4 KB per softmax warp
  static constexpr int kOnes = kOut + (RAGGED ? 0 : 2 * kBox);
  static constexpr int kBias = kOnes + 4096;
  static constexpr int kBar = kBias + kStages * 4096;
  // q_full[2], q_empty[2], k_full[S], k_empty[S], v_full[S], v_empty[S],
  // per box: s_full, s_empty, p_full, p_empty, o_full, o_empty; drain[3], never
  static constexpr int kNumBars = 4 + 4 * kStages + 2 * 6 + 4;
  static constexpr int kMisc = kBar + kNumBars * 8;
  static constexpr int kGeom = kMisc + 16;  // ragged mode: one geometry per warp
  static constexpr int kSmem = kGeom + (RAGGED ? (kThreadsF / 32) * (int)sizeof(Geom) : 0) + 1024;
  static_assert(kGeom % 8 == 0, "the geometries are copied in 8-byte words");
};
__device__ __forceinline__ uint32_t col_s(int x) { return 128u * x; }
__device__ __forceinline__ uint32_t col_p(int x) { return 256u + 64u * x; }
__device__ __forceinline__ uint32_t col_o(int x) { return 384u + 64u * x; }

struct Fwd64Args {
  Geom g;
  void* out;
  float* lse2;
  int items;  // B*nh * ntiles * box pairs
  uint32_t flags;
  int pad_R;  // box rows of every geometry of the launch (rows pad_R..127 of each block are zeroed once)
  // ragged mode (serving): per-request descriptors and device-side counts
  const ReqDesc* reqs;
  const int64_t* counts;
};

// One work item: a (batch*head, tile, pair of query boxes) of a geometry.
struct Item {
  const Geom* g;
  const CUtensorMap* tq;
  const CUtensorMap* tk;
  const CUtensorMap* tv;
  void* out;
  float* lse2;  // null in ragged mode, which stores none
  float* ot;    // ragged mode (else the slots' tensor map serves)
  int bh, tile, pair;
  int req;  // request index (ragged mode), else -1
};

inline int box_pairs(const Geom& g) { return (int)g.fpairs.d; }

// Ragged mode: the request that a warp's current item belongs to.  The search
// runs, and the request's geometry is copied into the warp's own block of
// shared memory, only when the item leaves the request's range: reading the
// geometry field by field from the descriptor table put a chain of global
// loads into every item of every role.
struct ReqCache {
  int req = -1, item0 = 0, item1 = 0;
  Geom* g = nullptr;  // the warp's block
};

// Returns false (after recording GATTN_ERR_DEVICE_BOUNDS) if a ragged work item
// does not decode to a valid (request, head, tile, pair); every role decodes
// the same item identically, so all of them skip it together.  SOLO: called by
// one lane of the warp, else by all of them together.
template <bool RAGGED, bool SOLO>
__device__ __forceinline__ bool resolve(const Fwd64Args& a, const CUtensorMap* tq, const CUtensorMap* tk,
                                        const CUtensorMap* tv, int w, ReqCache& rc, Item& it) {
  if constexpr (RAGGED) {
    if (w < rc.item0 || w >= rc.item1) {
      // requests are sorted by item0: binary search for the last item0 <= w
      const int nreq = (int)a.counts[0];
      int lo = 0, hi = nreq - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.reqs[mid].item0 <= w) lo = mid;
        else hi = mid - 1;
      }
      if (nreq < 1 || w < a.reqs[lo].item0 || w >= a.reqs[lo].item0 + a.reqs[lo].items) {
        set_status(kStatusBounds);
        return false;
      }
      rc.req = lo;
      rc.item0 = a.reqs[lo].item0;
      rc.item1 = rc.item0 + a.reqs[lo].items;
      static_assert(sizeof(Geom) % 8 == 0, "copied in 8-byte words");
      const uint64_t* src = reinterpret_cast<const uint64_t*>(&a.reqs[lo].g);
      uint64_t* dst = reinterpret_cast<uint64_t*>(rc.g);
      if constexpr (!SOLO) __syncwarp();
      for (int i = SOLO ? 0 : (threadIdx.x & 31); i < (int)(sizeof(Geom) / 8); i += SOLO ? 1 : 32) dst[i] = src[i];
      if constexpr (!SOLO) __syncwarp();
    }
    const ReqDesc& r = a.reqs[rc.req];
    it.g = rc.g;
    it.tq = it.tk = it.tv = &r.tmap;
    it.out = r.out;
    it.lse2 = nullptr;
    it.ot = r.ot;
    it.req = rc.req;
    w -= rc.item0;
  } else {
    it.g = &a.g;
    it.tq = tq;
    it.tk = tk;
    it.tv = tv;
    it.out = a.out;
    it.lse2 = a.lse2;
    it.ot = nullptr;
    it.req = -1;
  }
  const Geom& g = *it.g;
  const int r = fdiv(w, g.fpairs);
  it.pair = w - r * (int)g.fpairs.d;
  it.bh = fdiv(r, g.fntiles);
  it.tile = r - it.bh * g.ntiles;
  if (RAGGED && (it.bh >= g.B * g.nh || g.d != kD || g.R != a.pad_R)) {
    set_status(kStatusBounds);
    return false;
  }
  return true;
}

// running max of 32 scores into 4 partial maxima (3-input max)
__device__ __forceinline__ void chunk_max(const uint32_t* r, float (&mx)[4]) {
#pragma unroll
  for (int i = 0; i < 32; i += 2)
    mx[(i >> 1) & 3] = fmax3(mx[(i >> 1) & 3], __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
}

// exp2 of 32 scores -> 16 BF16 pairs, row sum in packed FP32 pairs
__device__ __forceinline__ void exp_chunk(const uint32_t* r, uint64_t s2, uint64_t nm2, uint64_t (&acc)[4],
                                          uint32_t (&pk)[16]) {
#pragma unroll
  for (int i = 0; i < 32; i += 2) {
    float a0, a1;
    f2unpack(ffma2(u2pack(r[i], r[i + 1]), s2, nm2), a0, a1);
    const float p0 = ex2(a0), p1 = ex2(a1);
    acc[(i >> 1) & 3] = fadd2(acc[(i >> 1) & 3], f2pack(p0, p1));
    pk[i >> 1] = pack_bf16(p0, p1);
  }
}

// multiply this thread's 64 O columns by f
__device__ __forceinline__ void rescale_o(uint32_t tO, float f) {
  const uint64_t f2 = f2pack(f, f);
  uint32_t r[32];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    tmem_ld32(tO + 32 * c, r);
    tmem_wait_ld(r);
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
      float x, y;
      f2unpack(fmul2(u2pack(r[i], r[i + 1]), f2), x, y);
      r[i] = __float_as_uint(x);
      r[i + 1] = __float_as_uint(y);
    }
    tmem_st32(tO + 32 * c, r);
  }
  tmem_wait_st();
}

// one output row of 64 FP32 values in registers, 16 bytes at a time
__device__ __forceinline__ void store_row(float* dst, const uint32_t (&r0)[32], const uint32_t (&r1)[32]) {
#pragma unroll
  for (int e = 0; e < 32; e += 4) {
    *reinterpret_cast<uint4*>(dst + e) = make_uint4(r0[e], r0[e + 1], r0[e + 2], r0[e + 3]);
    *reinterpret_cast<uint4*>(dst + 32 + e) = make_uint4(r1[e], r1[e + 1], r1[e + 2], r1[e + 3]);
  }
}
__device__ __forceinline__ void store_row(__nv_bfloat16* dst, const uint32_t (&r0)[32], const uint32_t (&r1)[32]) {
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const uint32_t* r = c == 0 ? r0 : r1;
#pragma unroll
    for (int e = 0; e < 32; e += 8)
      *reinterpret_cast<uint4*>(dst + 32 * c + e) =
          make_uint4(pack_bf16(__uint_as_float(r[e]), __uint_as_float(r[e + 1])),
                     pack_bf16(__uint_as_float(r[e + 2]), __uint_as_float(r[e + 3])),
                     pack_bf16(__uint_as_float(r[e + 4]), __uint_as_float(r[e + 5])),
                     pack_bf16(__uint_as_float(r[e + 6]), __uint_as_float(r[e + 7])));
  }
}

template <typename OutT, bool RAGGED>
__global__ void __launch_bounds__(kThreadsF, 1)
    fwd64_kernel(const __grid_constant__ CUtensorMap tq, const __grid_constant__ CUtensorMap tk,
                 const __grid_constant__ CUtensorMap tv, const __grid_constant__ CUtensorMap to,
                 const Fwd64Args a) {
  using C = Cfg<RAGGED>;
  constexpr int kStages = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kBar);
  uint64_t* q_full = bars;       // [2]
  uint64_t* q_empty = bars + 2;  // [2]
  uint64_t* k_full = bars + 4;
  uint64_t* k_empty = k_full + kStages;
  uint64_t* v_full = k_empty + kStages;
  uint64_t* v_empty = v_full + kStages;
  uint64_t* boxbar = v_empty + kStages;  // [x * 6 + i]
  auto s_full = [&](int x) { return boxbar + 6 * x; };
  auto s_empty = [&](int x) { return boxbar + 6 * x + 1; };
  auto p_full = [&](int x) { return boxbar + 6 * x + 2; };
  auto p_empty = [&](int x) { return boxbar + 6 * x + 3; };
  auto o_full = [&](int x) { return boxbar + 6 * x + 4; };
  auto o_empty = [&](int x) { return boxbar + 6 * x + 5; };
  uint64_t* drain = boxbar + 12;  // [3], one per issuing thread
  uint64_t* never = drain + 3;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::kMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::kMisc + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  zero_pad_rows(smem, 4 + 2 * kStages, a.pad_R);  // both Q buffers, the K and V rings
  // the ones operand (1 in K-column 0 of each of its 128 rows) and the zero
  // K-columns 8..15 of it and of every bias stage
  for (int r = threadIdx.x; r < (1 + kStages) * 256; r += kThreadsF) {
    const int blk = r >> 8, rr = r & 255;
    const uint4 v = (blk == 0 && rr < 128) ? make_uint4(0x00003F80u, 0u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
    if (blk == 0 || rr >= 128) *reinterpret_cast<uint4*>(smem + C::kOnes + blk * 4096 + rr * 16) = v;
  }
  fence_proxy_async_smem();
  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(q_full + b, 1);
      mbar_init(q_empty + b, RAGGED ? 1 : 1 + 8);  // the last score product; the softmax warps (staged outputs read)
    }
    for (int s = 0; s < kStages; ++s) {
      mbar_init(k_full + s, 1);
      mbar_init(k_empty + s, 1);
      mbar_init(v_full + s, 1);
      mbar_init(v_empty + s, 2);  // the P V product of each box
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(s_full(x), 1);
      mbar_init(s_empty(x), 4);
      mbar_init(p_full(x), 4);
      mbar_init(p_empty(x), 1);
      mbar_init(o_full(x), 1);
      mbar_init(o_empty(x), 4);
    }
    for (int i = 0; i < 3; ++i) mbar_init(drain + i, 1);
    mbar_init(never, 1);
    *abort_flag = 0;
    fence_mbar_init();
    if (!RAGGED) {
      prefetch_tmap(&tq);
      prefetch_tmap(&tk);
      prefetch_tmap(&tv);
      prefetch_tmap(&to);
    }
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int n_items = RAGGED ? (int)a.counts[1] : a.items;
  ReqCache rc;
  if constexpr (RAGGED) rc.g = reinterpret_cast<Geom*>(smem + C::kGeom) + warp;

  if (warp < kSoft0) {
    setmaxnreg_dec<kRegsLow>();
    if (warp == 0) {
      // ---------------------------------------------------------- TMA producer (lane 0) and key-mask writer
      // The whole warp walks the blocks: its lanes write the bias row of a block that has one, lane 0 does the
      // waits and the loads.  The arrival that announces K_j's load follows the row, so k_full covers both.
      const uint32_t neg = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(-1e30f));
      uint32_t G = 0, W = 0;
      uint32_t q_arm = 0, q_par = 0, k_arm = 0, k_par = 0, v_arm = 0, v_par = 0;  // lane 0's
      int last_req = -1;
      bool ok = true;
      auto all_ok = [&]() { return ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0; };
      for (int w = blockIdx.x; w < n_items && ok; w += gridDim.x) {
        Item it;
        if (!resolve<RAGGED, false>(a, &tq, &tk, &tv, w, rc, it)) continue;
        const Geom& g = *it.g;
        const int bh = it.bh;
        TileBlocks tbk;
        tile_blocks(g, it.tile, tbk);
        const int qa = 2 * it.pair;
        if (qa >= tbk.NB) continue;
        const int nact = qa + 1 < tbk.NB ? 2 : 1;
        if (lane == 0) {
          if (RAGGED && it.req != last_req) {
            tmap_acquire(it.tq);  // this launch's descriptor table may hold a new map here
            last_req = it.req;
          }
          // Q of this item goes to buffer W & 1, so it loads while the previous
          // item's score products still read the other buffer
          const uint32_t qb = W & 1, qn = (W >> 1) & 1;
          if ((ok = WAIT(q_empty + qb, qn ^ 1))) {
            mbar_arrive_expect_tx(q_full + qb, nact * g.R * 128);
            q_arm |= 1u << qb;
            q_par = (q_par & ~(1u << qb)) | (qn << qb);
            for (int x = 0; x < nact; ++x) {
              int o[3];
              block_origin(g, tbk, qa + x, o);
              tma_load_5d(smem + C::kQ + (2 * qb + x) * kBox, it.tq, q_full + qb, 0, tbk.tb.lo[2] + o[2],
                          tbk.tb.lo[1] + o[1], tbk.tb.lo[0] + o[0], bh);
            }
          }
        }
        const bool all_full = tile_all_full(g, tbk);
        BlockWalk bw;
        for (int j = 0; j < tbk.NB; ++j, ++G, bw.next(tbk)) {
          const uint32_t st = G % kStages, n = G / kStages;
          const int ko[3] = {bw.jt * g.bt, bw.jy * g.by, bw.jx * g.bx};
          if (lane == 0 && ok) ok = WAIT(k_empty + st, (n & 1) ^ 1);
          if (!all_ok()) break;
          if (!all_full && !bw.full(g, tbk)) {
            for (int r = lane; r < 128; r += 32) {
              int kl[3];
              block_row(g, ko, r, kl);
              *reinterpret_cast<uint4*>(smem + C::kBias + st * 4096 + r * 16) =
                  make_uint4(inside(tbk, kl) ? 0u : neg, 0u, 0u, 0u);
            }
            fence_proxy_async_smem();  // the tensor core reads what these lanes wrote
            __syncwarp();
          }
          if (lane == 0) {
            const int c1 = tbk.tb.lo[2] + ko[2], c2 = tbk.tb.lo[1] + ko[1], c3 = tbk.tb.lo[0] + ko[0];
            mbar_arrive_expect_tx(k_full + st, g.R * 128);
            k_arm |= 1u << st;
            k_par = (k_par & ~(1u << st)) | ((n & 1) << st);
            tma_load_5d(smem + C::kK + st * kBox, it.tk, k_full + st, 0, c1, c2, c3, bh);
            if ((ok = WAIT(v_empty + st, (n & 1) ^ 1))) {
              mbar_arrive_expect_tx(v_full + st, g.R * 128);
              v_arm |= 1u << st;
              v_par = (v_par & ~(1u << st)) | ((n & 1) << st);
              tma_load_5d(smem + C::kV + st * kBox, it.tv, v_full + st, 0, c1, c2, c3, bh);
            }
          }
        }
        if (!all_ok()) break;
        ++W;
      }
      if (!ok && lane == 0) {
        // let every load this thread issued land before the CTA exits
        for (int b = 0; b < 2; ++b)
          if (q_arm & (1u << b)) mbar_wait<set_status_f64>(q_full + b, (q_par >> b) & 1, abort_flag, false);
        for (int s = 0; s < kStages; ++s) {
          if (k_arm & (1u << s)) mbar_wait<set_status_f64>(k_full + s, (k_par >> s) & 1, abort_flag, false);
          if (v_arm & (1u << s)) mbar_wait<set_status_f64>(v_full + s, (v_par >> s) & 1, abort_flag, false);
        }
      }
    } else if (warp == 1 && lane == 0) {
      // ---------------------------------------------------------- issuer of S_x = Q_x K^T
      constexpr uint32_t idS = idesc_bf16(128, 128, 0);
      const uint64_t dQ0 = sw128_desc(smem_u32(smem + C::kQ), 16, 1024);
      const uint64_t dK0 = sw128_desc(smem_u32(smem + C::kK), 16, 1024);
      const uint64_t dOnes = noswz_desc(smem_u32(smem + C::kOnes), 2048, 128);
      const uint64_t dBias0 = noswz_desc(smem_u32(smem + C::kBias), 2048, 128);
      uint32_t G = 0, W = 0, GX0 = 0, GX1 = 0;
      bool ok = true;
      if (a.flags & GATTN_FLAG_TEST_STALL)  // failure-detection hook: a wait that cannot complete
        ok = mbar_wait<set_status_f64>(never, 0, abort_flag, true, 20000000ull);
      for (int w = blockIdx.x; w < n_items && ok; w += gridDim.x) {
        Item it;
        if (!resolve<RAGGED, true>(a, &tq, &tk, &tv, w, rc, it)) continue;
        const Geom& g = *it.g;
        TileBlocks tbk;
        tile_blocks(g, it.tile, tbk);
        const int qa = 2 * it.pair;
        if (qa >= tbk.NB) continue;
        const int nact = qa + 1 < tbk.NB ? 2 : 1;
        const uint32_t qb = W & 1;
        if (!(ok = WAIT(q_full + qb, (W >> 1) & 1))) break;  // Q_A, Q_B of this item in shared memory
        const bool all_full = tile_all_full(g, tbk);
        BlockWalk bw;
        for (int j = 0; j < tbk.NB && ok; ++j, ++G, bw.next(tbk)) {
          const uint32_t st = G % kStages;
          // a masked block's bias row was written by the producer warp
          const bool masked = !all_full && !bw.full(g, tbk);
          if (!(ok = WAIT(k_full + st, (G / kStages) & 1))) break;
          const uint64_t dk = dmove(dK0, st * kBox), db = dmove(dBias0, st * 4096);
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            if (x >= nact) break;
            uint32_t& gx = x == 0 ? GX0 : GX1;
            // S_x is free once the softmax threads have read the previous scores
            if (gx > 0 && !(ok = WAIT(s_empty(x), (gx - 1) & 1))) break;
            tc_fence_after();
            const uint64_t dq = dmove(dQ0, (2 * qb + x) * kBox);
#pragma unroll
            for (int ks = 0; ks < kD / 16; ++ks)
              umma_bf16(tmem + col_s(x), dmove(dq, ks * 32), dmove(dk, ks * 32), idS, ks > 0);
            if (masked) umma_bf16(tmem + col_s(x), dOnes, db, idS, 1u);  // + bias of each key column
            umma_commit(s_full(x));
            ++gx;
          }
          if (!ok) break;
          umma_commit(k_empty + st);
        }
        if (!ok) break;
        umma_commit(q_empty + qb);  // Q_A, Q_B of this item no longer read
        ++W;
      }
      umma_commit(drain);
      mbar_wait<set_status_f64>(drain, 0, abort_flag, false);
    } else if (warp >= 2 && lane == 0) {
      // ---------------------------------------------------------- issuers of O_x += P_x V, one thread per box
      const int x = warp - 2;
      constexpr uint32_t idO = idesc_bf16(128, kD, 1);
      const uint64_t dV0 = sw128_desc(smem_u32(smem + C::kV), 16384, 1024);  // MN-major (K = keys)
      const uint32_t tO = tmem + col_o(x), tP = tmem + col_p(x);
      uint32_t G = 0, GX = 0, WX = 0;
      bool ok = true;
      for (int w = blockIdx.x; w < n_items && ok; w += gridDim.x) {
        Item it;
        if (!resolve<RAGGED, true>(a, &tq, &tk, &tv, w, rc, it)) continue;
        TileBlocks tbk;
        tile_blocks(*it.g, it.tile, tbk);
        const int qa = 2 * it.pair;
        if (qa >= tbk.NB) continue;
        const bool act = qa + x < tbk.NB;
        for (int j = 0; j < tbk.NB; ++j, ++G) {
          const uint32_t st = G % kStages;
          if (!(ok = WAIT(v_full + st, (G / kStages) & 1))) break;
          if (!act) {  // an item of one box: the other issuer's product is V_j's only reader
            mbar_arrive(v_empty + st);
            continue;
          }
          const uint64_t dv = dmove(dV0, st * kBox);
          if (!(ok = WAIT(p_full(x), GX & 1))) break;
          if (j == 0 && !(ok = WAIT(o_empty(x), (WX & 1) ^ 1))) break;
          tc_fence_after();
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)
            umma_bf16_ts(tO, tP + ks * 8, dmove(dv, ks * 2048), idO, (j > 0 || ks > 0) ? 1u : 0u);
          umma_commit(p_empty(x));
          if (j == tbk.NB - 1) umma_commit(o_full(x));
          umma_commit(v_empty + st);
          ++GX;
        }
        if (act) ++WX;
      }
      umma_commit(drain + 1 + x);
      mbar_wait<set_status_f64>(drain + 1 + x, 0, abort_flag, false);
    }
  } else {
    setmaxnreg_inc<kRegsHigh>();
    // ------------------------------------------------------------ softmax + epilogue of box x
    const int x = (warp - kSoft0) >> 2;
    const int quad = warp & 3;
    const int row = quad * 32 + lane;  // TMEM lane = query row of the box
    const uint32_t tl = tmem + ((uint32_t)(quad * 32) << 16);
    const uint32_t tS = tl + col_s(x), tP = tl + col_p(x), tO = tl + col_o(x);
    // this warp's staging blocks: 32 rows x 128 bytes of the output row's columns 0..31
    // (its rows of the item's own Q block, which the score products are done with) and 32..63
    const uint32_t st_q = smem_u32(smem + C::kQ) + x * kBox + quad * 4096;
    const uint32_t st_o = smem_u32(smem + C::kOut) + (warp - kSoft0) * 4096;
    uint32_t GX = 0, WX = 0, W = 0;
    int staged = -1;  // Q buffer whose staged output may still be read by this warp's stores
    bool ok = true;
    // the stores have read the staged rows: the Q buffer may be refilled
    auto release_staged = [&]() {
      if (staged >= 0 && lane == 0) {
        bulk_wait_read();
        mbar_arrive(q_empty + staged);
      }
      staged = -1;
    };
    for (int w = blockIdx.x; w < n_items && ok; w += gridDim.x) {
      Item it;
      if (!resolve<RAGGED, false>(a, &tq, &tk, &tv, w, rc, it)) continue;
      const Geom& g = *it.g;
      const int bh = it.bh, tile = it.tile;
      const float sl2 = g.scale_log2;
      const uint64_t s2 = f2pack(sl2, sl2);
      TileBlocks tbk;
      tile_blocks(g, it.tile, tbk);
      const int qa = 2 * it.pair;
      if (qa >= tbk.NB) continue;
      const uint32_t buf = W & 1;
      if (qa + x >= tbk.NB) {  // an item of one box: this warp only passes its Q buffer on
        if constexpr (!RAGGED) {
          release_staged();
          if (!(ok = WAIT(q_full + buf, (W >> 1) & 1))) break;
          if (lane == 0) mbar_arrive(q_empty + buf);
          ++W;
        }
        continue;
      }
      const int nb = tbk.NB;
      // ragged mode resolves the row's place before its key blocks and keeps it,
      // the other mode resolves it again after them (see the epilogue)
      const int qb = qa + x;
      int ql[3] = {0, 0, 0};
      bool qvalid = false;
      if constexpr (RAGGED) {
        int qo[3];
        block_origin(g, tbk, qb, qo);
        block_row(g, qo, row, ql);
        qvalid = inside(tbk, ql);
      }
      float m = -INFINITY, l = 0.f, lc = 0.f;  // lc: Kahan compensation of the row sum l
      bool s_ready = false;
      for (int j = 0; j < nb; ++j, ++GX) {
        if (!s_ready && !(ok = WAIT(s_full(x), GX & 1))) break;
        tc_fence_after();
        // the row's 128 scores into registers, then S_x is released
        uint32_t s0[32], s1[32], s2r[32], s3[32];
        tmem_ld32(tS, s0);
        tmem_ld32(tS + 32, s1);
        tmem_ld32(tS + 64, s2r);
        tmem_ld32(tS + 96, s3);
        tmem_wait_ld(s0);
        tmem_wait_ld(s1);
        tmem_wait_ld(s2r);
        tmem_wait_ld(s3);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(s_empty(x));
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
        // masked keys carry -1e30 from the extension step: no mask here
        chunk_max(s0, mx);
        chunk_max(s1, mx);
        chunk_max(s2r, mx);
        chunk_max(s3, mx);
        const float mblk = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sl2;
        float f = 1.f;
        bool any_grow = false;
        if (j == 0) {
          m = mblk;
        } else {
          const bool grow = mblk > m + kRescaleLog2;
          any_grow = __any_sync(0xffffffffu, grow);
          if (grow) {
            f = ex2(m - mblk);
            m = mblk;
          }
        }
        // the exponentials depend only on the scores and the new reference max:
        // they are computed into registers before P_x is known to be free
        const uint64_t nm2 = f2pack(-m, -m);
        uint64_t acc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = f2pack(0.f, 0.f);
        uint32_t pk0[16], pk1[16], pk2[16], pk3[16];
        exp_chunk(s0, s2, nm2, acc, pk0);
        exp_chunk(s1, s2, nm2, acc, pk1);
        exp_chunk(s2r, s2, nm2, acc, pk2);
        exp_chunk(s3, s2, nm2, acc, pk3);
        float lsum = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float u, v;
          f2unpack(acc[i], u, v);
          lsum += u + v;
        }
        // P_x and O_x are free once the previous P V of this box completed
        if (GX > 0 && !(ok = WAIT(p_empty(x), (GX - 1) & 1))) break;
        tc_fence_after();
        if (any_grow) {
          rescale_o(tO, f);
          l *= f;
          lc *= f;
        }
        {  // compensated sum over the tile's key blocks
          const float y = lsum - lc;
          const float t = l + y;
          lc = (t - l) - y;
          l = t;
        }
        tmem_st16(tP, pk0);
        tmem_st16(tP + 16, pk1);
        tmem_st16(tP + 32, pk2);
        tmem_st16(tP + 48, pk3);
        // the next scores are usually there by now: ask while P is being stored (tiles
        // of 36864 tokens 59.7 -> 58.4 ms; ragged mode is 1 % slower with it)
        s_ready = !RAGGED && j + 1 < nb && mbar_try_wait(smem_u32(s_full(x)), (GX + 1) & 1);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(p_full(x));
        if (!RAGGED && j == 0) release_staged();  // the previous item's stores have had this block's time
      }
      if (!ok) break;
      // ---- epilogue: wait for the last P V, O / l.  Two forms, because ptxas's
      // schedule of the softmax loop above hangs on what stays live across it
      // (the same loop ran between 57 and 84 ms on the paper-regime tiles):
      //   one problem: the row's place is resolved here, while the last P V runs,
      //     and slots leave by TMA (small tiles 2.15 -> 2.01 ms)
      //   ragged: resolved before the loop, plain stores (each request has its own
      //     tensor map, which every storing warp would have to acquire; 3.21 ms per
      //     iteration of six requests, 3.7 in the other form)
      if constexpr (RAGGED) {
        if (!(ok = WAIT(o_full(x), WX & 1))) break;
        tc_fence_after();
        ++WX;
        const float inv = 1.f / l;
        const int64_t slot = tile_slot0(g, bh, tile) + qb * 128 + row;
        const int p[3] = {tbk.tb.lo[0] + ql[0], tbk.tb.lo[1] + ql[1], tbk.tb.lo[2] + ql[2]};
        const int64_t tok = qvalid ? ((int64_t)p[0] * g.G[1] + p[1]) * g.G[2] + p[2] : 0;
        const bool single = qvalid && only_cover(g, tbk.tb, p);
        OutT* dst_out = static_cast<OutT*>(it.out) + ((int64_t)bh * g.N + tok) * kD;
        float* dst_scr = it.ot + slot * kD;
        // the whole O row into registers, then O_x is released at once: the next
        // item's first P V may overwrite it while this row is scaled and stored
        uint32_t r0[32], r1[32];
        tmem_ld32(tO, r0);
        tmem_ld32(tO + 32, r1);
        tmem_wait_ld(r0);
        tmem_wait_ld(r1);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(o_empty(x));
        if (qvalid) {
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const uint32_t* r = c == 0 ? r0 : r1;
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              const float4 v4 = make_float4(__uint_as_float(r[e]) * inv, __uint_as_float(r[e + 1]) * inv,
                                            __uint_as_float(r[e + 2]) * inv, __uint_as_float(r[e + 3]) * inv);
              if (single)
                store4<OutT>(dst_out + c * 32 + e, v4);
              else
                store4<float>(dst_scr + c * 32 + e, v4);
            }
          }
        }
      } else {
        Item it2;
        TileBlocks tb2;
        resolve<RAGGED, false>(a, &tq, &tk, &tv, w, rc, it2);
        const Geom& g2 = *it2.g;
        tile_blocks(g2, it2.tile, tb2);
        const int qb2 = 2 * it2.pair + x;
        int qo[3], l2[3];
        block_origin(g2, tb2, qb2, qo);
        block_row(g2, qo, row, l2);
        const bool valid = inside(tb2, l2);
        const float inv = 1.f / l;
        const int64_t slot = tile_slot0(g2, it2.bh, it2.tile) + qb2 * 128 + row;
        if (valid) it2.lse2[slot] = m + __log2f(l);
        const int p[3] = {tb2.tb.lo[0] + l2[0], tb2.tb.lo[1] + l2[1], tb2.tb.lo[2] + l2[2]};
        const int64_t tok = valid ? ((int64_t)p[0] * g2.G[1] + p[1]) * g2.G[2] + p[2] : 0;
        const bool single = valid && only_cover(g2, tb2.tb, p);
        if (!(ok = WAIT(o_full(x), WX & 1))) break;
        tc_fence_after();
        ++WX;
        uint32_t r0[32], r1[32];
        tmem_ld32(tO, r0);
        tmem_ld32(tO + 32, r1);
        tmem_wait_ld(r0);
        tmem_wait_ld(r1);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(o_empty(x));
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          r0[e] = __float_as_uint(__uint_as_float(r0[e]) * inv);
          r1[e] = __float_as_uint(__uint_as_float(r1[e]) * inv);
        }
        if (single) store_row(static_cast<OutT*>(it2.out) + ((int64_t)it2.bh * g2.N + tok) * kD, r0, r1);
        if (__any_sync(0xffffffffu, valid && !single)) {
          // FP32 slots of this warp's 32 rows, through shared memory (rows past R
          // stay zero, they are padding of the Q block; slots of rows that are
          // not multiply covered are never read)
          const uint32_t sq = st_q + buf * 2 * kBox;
          if (row < a.pad_R) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const uint32_t off = lane * 128 + ((c ^ (lane & 7)) << 4);
              st_shared_v4(sq + off, r0[4 * c], r0[4 * c + 1], r0[4 * c + 2], r0[4 * c + 3]);
              st_shared_v4(st_o + off, r1[4 * c], r1[4 * c + 1], r1[4 * c + 2], r1[4 * c + 3]);
            }
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            const int srow = (int)(slot - lane);
            tma_store_2d(&to, sq, 0, srow);
            tma_store_2d(&to, st_o, 32, srow);
            bulk_commit();
          }
        }
        staged = (int)buf;
        ++W;
      }
    }
    release_staged();
    if (lane == 0) bulk_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

template <typename OutT>
cudaError_t run_fwd64(const Geom& g, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                      void* out, float* lse2, float* ot, uint32_t flags, cudaStream_t st) {
  Fwd64Args a;
  memset(&a, 0, sizeof(a));
  a.g = g;
  a.out = out;
  a.lse2 = lse2;
  a.flags = flags;
  a.pad_R = g.R;
  const int64_t items = (int64_t)g.B * g.nh * g.ntiles * box_pairs(g);
  if (items >= (1LL << 31)) return cudaErrorNotSupported;
  a.items = (int)items;
  const int BH = g.B * g.nh;
  CUtensorMap mq, mk, mv, mo;
  if (!make_tmap_5d(&mq, q, kD, g.G[2], g.G[1], g.G[0], BH, g.bx, g.by, g.bt) ||
      !make_tmap_5d(&mk, k, kD, g.G[2], g.G[1], g.G[0], BH, g.bx, g.by, g.bt) ||
      !make_tmap_5d(&mv, v, kD, g.G[2], g.G[1], g.G[0], BH, g.bx, g.by, g.bt) ||
      !make_tmap_slots(&mo, ot, kD, (int64_t)BH * g.ntiles * g.per_tile, 32))
    return cudaErrorInvalidValue;
  auto kern = fwd64_kernel<OutT, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<false>::kSmem);
  if (e != cudaSuccess) return e;
  const int grid = (int)(a.items < num_sms() ? a.items : num_sms());
  kern<<<grid, kThreadsF, Cfg<false>::kSmem, st>>>(mq, mk, mv, mo, a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sm103_fwd64(const Geom& g, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                               void* out, int out_dtype, float* lse2, float* ot, uint32_t flags, cudaStream_t st) {
  if (g.d != kD) return cudaErrorNotSupported;
  if (out_dtype == GATTN_BF16) return run_fwd64<__nv_bfloat16>(g, q, k, v, out, lse2, ot, flags, st);
  return run_fwd64<float>(g, q, k, v, out, lse2, ot, flags, st);
}

int fwd64_ragged_items(const Geom& g) { return g.nh * g.ntiles * box_pairs(g); }

cudaError_t launch_sm103_fwd64_ragged(const ReqDesc* reqs, const int64_t* counts, int box_rows, cudaStream_t st) {
  Fwd64Args a;
  memset(&a, 0, sizeof(a));
  a.reqs = reqs;
  a.counts = counts;
  a.pad_R = box_rows;
  CUtensorMap dummy;
  memset(&dummy, 0, sizeof(dummy));
  auto kern = fwd64_kernel<__nv_bfloat16, true>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<true>::kSmem);
  if (e != cudaSuccess) return e;
  kern<<<num_sms(), kThreadsF, Cfg<true>::kSmem, st>>>(dummy, dummy, dummy, dummy, a);
  return cudaGetLastError();
}

}  // namespace gattn
