// Attention over the full spatio-temporal token sequence (self, joint and
// cross attention of the DiT blocks).  RoPE is applied to q and k once per
// token by the QKV projection's epilogue, so this kernel reads pre-rotated
// operands.
//
// bf16 path: a flash-attention kernel on tcgen05 tensor cores.  A work item
// is two 128-row query tiles (a, b) of one head; its CTA streams K/V tiles (128
// keys; 64 for short ranges at head dim 64) that both query tiles share:
//   warp 0      TMA producer: Q_a, Q_b once per item, K_j and V_j into rings
//               (128-byte swizzle);
//   warp 1      MMA issuer: S_t = Q_t K_j^T lands in a region of TMEM, P_t is
//               written back over it (bf16, two per column) and O_t += P_t V_j
//               reads P_t from TMEM and V_j from shared memory.  The tiles
//               alternate, and each PV is followed by the S that takes its
//               region over, so that the tensor core works on one query tile
//               while the softmax of the other runs;
//   warps 2-5   softmax of tile a, warps 6-9 softmax of tile b: one thread
//               per query row keeps the running max and sum, and rescales O_t
//               in TMEM only when the running max grows by more than 2^8 (the
//               final division by the sum makes the result independent of
//               when rescaling happens).
// attn_persist_kernel runs whole items on persistent CTAs: the next item's Q
// loads and first S MMAs overlap the current item's last softmax, and the
// output leaves through shared memory and TMA stores.  attn_split_kernel runs
// the items of a partial last wave, each split along its key range over
// several CTAs, and attn_merge_kernel puts their parts together.
// fp32 path: attn_f32_kernel, a tiled flash kernel on the FP32 pipes with exact
// expf, for the fp32 mode.
#include <cudaTypedefs.h>
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace acid {

acid_status make_tmap_bf16(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows);
acid_status make_tmap_bf16_box(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld,
                               int box_cols, int box_rows, CUtensorMapSwizzle swizzle);

namespace {

constexpr int kTileQ = 128;  // query rows per tile (two tiles per CTA)
constexpr int kBQ = 2 * kTileQ;
constexpr int kAttnThreads = 320;
constexpr float kRescaleLog2 = 8.0f, kRescale = 256.0f;
constexpr int kAttnPartCtas = kAttnSplitCtas;  // CTAs of a split tail wave (partials workspace capacity)

struct AttnDev {
  int64_t nq, nk;
  int q_col, k_col, v_col;
  void* out;
  int64_t ldo;
  int o_col;
  float scale_log2;  // log2(e) / sqrt(head_dim)
  // work item = (query-tile pair, head), numbered head-major.  attn_split_kernel:
  // CTA blockIdx.x handles item item_base + blockIdx.x / splits and the
  // split-th part of the key range, and writes its unnormalised output and
  // (max, sum) per row to part_o / part_ml.  attn_persist_kernel: CTA blockIdx.x
  // handles items item_base + blockIdx.x + k * gridDim.x below item_end.
  int nqp;
  int item_base, item_end;
  int splits;
  float* part_o;   // [CTA][256 rows][D]
  float* part_ml;  // [CTA][256 rows][2]
};

// Head dim and keys per K/V tile of a kernel.
template <int HEAD_DIM, int KEYS>
struct AttnCfg {
  static constexpr int D = HEAD_DIM, BKV = KEYS;
  // S regions in TMEM.  Step n of a CTA (2 * key-tile step + query tile: the
  // tiles alternate) uses region n % NB, and S(n + NB) is issued right after
  // PV(n), which reads P(n) from it.  Head dim 128: S and O of both query tiles
  // fill TMEM.  Head dim 64: O needs half the columns, and a third region lets
  // the tensor cores run ahead of the softmax warps, which set the pace at this
  // head dim: a step costs them about 630 clocks whatever its keys and 9.4 more
  // per key (4726 tokens, 30 heads: 197.6 us in 64-key tiles on four regions,
  // 163.1 in 96-key tiles on four, 146.6 in 128-key tiles on these three).
  // 64-key tiles are for the shortest key ranges, where starting and ending
  // items weighs most: 256 columns, two CTAs on an SM.
  static constexpr int CTAS_PER_SM = BKV == 64 ? 2 : 1;
  static constexpr int NB = D <= 64 && BKV == 128 ? 3 : 2;
  static constexpr int KVS = NB == 3 ? 4 : 2;        // K and V ring depth
  // Whether a tile's row max is formed before its exponentials or only where the
  // row sum asks for it (softmax_tile).  At head dim 128 the MMAs and power set
  // the pace and the two take the same time; two CTAs on an SM leave too few
  // registers to keep a row until its sum is known.
  static constexpr bool MAX_FIRST = !(D == 64 && BKV == 128);
  static constexpr int CH = D / 64;                  // 64-column chunks per row
  static constexpr int CHUNK_Q = 128 * 128;          // 128 rows x 128 bytes
  static constexpr int CHUNK_KV = BKV * 128;         // BKV rows x 128 bytes
  static constexpr int T_BYTES = CH * CHUNK_Q;       // one 128-row tile of Q
  static constexpr int KV_BYTES = CH * CHUNK_KV;     // one K or V tile
  static constexpr int OFF_Q = 0;                    // Q_a, Q_b
  static constexpr int OFF_K = OFF_Q + 2 * T_BYTES;  // rings
  static constexpr int OFF_V = OFF_K + KVS * KV_BYTES;
  static constexpr int OFF_BAR = OFF_V + KVS * KV_BYTES;
  static constexpr int BAR_BYTES = 512;
  static constexpr int SMEM = OFF_BAR + BAR_BYTES + 1024;
  // attn_persist_kernel adds the output staging: per softmax warp two
  // 32-row x 32-column bf16 boxes (64-byte swizzle) for TMA stores
  static constexpr int STAGE_BOX = 32 * 64;
  static constexpr int OFF_STAGE_P = OFF_V + KVS * KV_BYTES;
  static constexpr int OFF_BAR_P = OFF_STAGE_P + 8 * 2 * STAGE_BOX;
  static constexpr int SMEM_P = OFF_BAR_P + BAR_BYTES + 1024;
  // TMEM columns: the S regions (P over the first BKV / 2 columns of each), O_a, O_b
  static constexpr uint32_t O_COL = NB * BKV, TMEM_COLS = O_COL + 2 * D;
  static_assert(TMEM_COLS * CTAS_PER_SM == 512, "the CTAs of an SM take all of TMEM");
  __host__ __device__ static constexpr uint32_t o_col(int t) { return O_COL + t * D; }
  // Region of step g of tile t, and the parity of its use.
  static __device__ __forceinline__ int sb(int t, int g) { return NB == 2 ? t : (2 * g + t) % NB; }
  static __device__ __forceinline__ uint32_t sp(int t, int g) { return (uint32_t)(NB == 2 ? g : (2 * g + t) / NB) & 1; }
  static __device__ __forceinline__ int slot(int g) { return g & (KVS - 1); }
  static __device__ __forceinline__ uint32_t round(int g) { return (uint32_t)(g / KVS); }
};

// The barriers of a CTA.
template <class C>
struct AttnBars {
  uint64_t *q_full, *q_empty;  // [2] per query tile
  uint64_t *k_full, *k_empty, *v_full, *v_empty;  // [KVS]
  uint64_t *s_full, *p_full, *pv_done;  // [NB] per S region
  uint64_t* drain;  // failure path: the MMAs issued so far have completed
  uint32_t* tmem_slot;
  static constexpr int kCount = 4 + 4 * C::KVS + 3 * C::NB + 1;
  static_assert(kCount * 8 + 4 <= C::BAR_BYTES, "barrier area");
  __device__ __forceinline__ explicit AttnBars(uint8_t* at) {
    uint64_t* b = reinterpret_cast<uint64_t*>(at);
    auto take = [&](int n) { uint64_t* r = b; b += n; return r; };
    q_full = take(2);
    q_empty = take(2);
    k_full = take(C::KVS);
    k_empty = take(C::KVS);
    v_full = take(C::KVS);
    v_empty = take(C::KVS);
    s_full = take(C::NB);
    p_full = take(C::NB);
    pv_done = take(C::NB);
    drain = take(1);
    tmem_slot = reinterpret_cast<uint32_t*>(b);
  }
  __device__ __forceinline__ void init() const {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&q_full[i], 1);
      mbar_init(&q_empty[i], 1);
    }
    for (int i = 0; i < C::KVS; ++i) {
      mbar_init(&k_full[i], 1);
      mbar_init(&k_empty[i], 1);
      mbar_init(&v_full[i], 1);
      mbar_init(&v_empty[i], 1);
    }
    for (int i = 0; i < C::NB; ++i) {
      mbar_init(&s_full[i], 1);
      mbar_init(&p_full[i], 128);
      mbar_init(&pv_done[i], 1);
    }
    mbar_init(drain, 1);
    mbar_fence_init();
  }
};

// Softmax of one key tile for this thread's query row (row r of tile t is
// TMEM lane r): waits for S_t, writes P_t = 2^(s * scale - m) over the S
// region as bf16 pairs, updates the running reference max m and sum l,
// rescales O_t when the reference moves, and hands P_t to the MMA warp.
// g: this tile's step count in the CTA; first: the item's first key tile;
// valid: keys of a masked (partial last) tile.
template <class C, bool MASKED>
__device__ __forceinline__ bool softmax_tile(const AttnBars<C>& bar, int t, int g, bool first, int valid,
                                             uint32_t s_base, uint32_t o_addr, float scale_log2, float& m_run,
                                             float& l_run) {
  const uint32_t s_addr = s_base + C::sb(t, g) * C::BKV;
  // The lanes of a warp wait on the same phase, so they give up together
  // (after the wait limit) and the warp-collective tcgen05.ld / st below stay
  // convergent; a vote here would rule out a phase that completes exactly at
  // the limit for some lanes only, but costs 2-3% in this loop.
  if (!mbar_wait(&bar.s_full[C::sb(t, g)], C::sp(t, g))) return false;
  tc_fence_after();
  float s[C::BKV];
#pragma unroll
  for (int c = 0; c < C::BKV / 32; ++c) tmem_ld32(s_addr + c * 32, reinterpret_cast<uint32_t*>(s + c * 32));
  tmem_wait_ld();
  bool resc = false;
  float f = 1.0f;
  if constexpr (MASKED) {
#pragma unroll
    for (int i = 0; i < C::BKV; ++i)
      if (i >= valid) s[i] = -INFINITY;
  }
  const uint64_t sc2 = f2_pack(scale_log2, scale_log2);
  const float mref = first ? 0.f : m_run;
  const uint64_t nm2 = f2_pack(-mref, -mref);
  auto row_max = [](const float* m4) { return fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])); };
  auto shift = [&](float me) {
    const uint64_t sh2 = f2_pack(-me, -me);
#pragma unroll
    for (int i = 0; i < C::BKV / 2; ++i)
      f2_unpack(f2_add(f2_pack(s[2 * i], s[2 * i + 1]), sh2), s[2 * i], s[2 * i + 1]);
  };
  // P = 2^e as bf16 pairs over the first BKV/2 columns of S_t, and the row sum
  // as packed fp32 pairs
  auto exps = [&]() -> float {
    uint64_t acc0 = f2_pack(0.f, 0.f), acc1 = acc0;
#pragma unroll
    for (int half = 0; half < C::BKV / 64; ++half) {
      uint32_t pk[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float p0 = ex2_approx(s[half * 64 + 2 * i]), p1 = ex2_approx(s[half * 64 + 2 * i + 1]);
        if (i & 1)
          acc1 = f2_add(acc1, f2_pack(p0, p1));
        else
          acc0 = f2_add(acc0, f2_pack(p0, p1));
        pk[i] = pack_bf16(p0, p1);
      }
      tmem_st32(s_addr + half * 32, pk);
    }
    float a0, a1, b0, b1;
    f2_unpack(acc0, a0, a1);
    f2_unpack(acc1, b0, b1);
    return (a0 + a1) + (b0 + b1);
  };
  // e = s * scale - m_run in place (packed pairs; the first tile uses 0 as the
  // reference); the row max of e in four independent 3-input max chains on the
  // ALU pipe.  The P_t region is free here: the MMAs run in order, and S_t(g)
  // follows the PV that read it.  Lazy rescaling: the reference max moves only
  // on the first tile or when the row max exceeds it by more than 2^8; then e
  // is shifted in place.
  float ls;
  if constexpr (C::MAX_FIRST) {
    float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int i = 0; i < C::BKV / 2; ++i) {
      f2_unpack(f2_fma(f2_pack(s[2 * i], s[2 * i + 1]), sc2, nm2), s[2 * i], s[2 * i + 1]);
      m4[i & 3] = fmax3(m4[i & 3], s[2 * i], s[2 * i + 1]);
    }
    const float me = row_max(m4);
    if (first || me > kRescaleLog2) {
      if (!first) {
        resc = true;
        f = ex2_approx(-me);
        l_run *= f;
      }
      m_run = mref + me;
      shift(me);
    }
    ls = exps();
  } else {
    // An element above 2^8 makes the row sum larger than 2^8 (or NaN), so the
    // max is formed on a row's first tile and then only for such a sum.  Where
    // it moves the reference, the warp writes its P again.  Without the max the
    // exponentials start as the scores are scaled: 4726 tokens, 30 heads 172.9 ->
    // 158.9 us (with 96-key tiles).  A row that moves at every tile pays its
    // exponentials twice: with scores that rise by 2^10 from tile to tile 290 us,
    // where the max first takes 207 to 228 (64-key tiles).  A flag that lets a
    // tile behind a move form its max first takes 211 there, but ordinary scores
    // 151 instead of 147 and peaked ones 171 instead of 162, so there is none.
    auto max_of_e = [&] {
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int i = 0; i < C::BKV / 2; ++i) m4[i & 3] = fmax3(m4[i & 3], s[2 * i], s[2 * i + 1]);
      return row_max(m4);
    };
#pragma unroll
    for (int i = 0; i < C::BKV / 2; ++i)
      f2_unpack(f2_fma(f2_pack(s[2 * i], s[2 * i + 1]), sc2, nm2), s[2 * i], s[2 * i + 1]);
    if (first) {
      m_run = max_of_e();
      shift(m_run);
    }
    ls = exps();
    if (!first && !(ls <= kRescale)) {
      const float me = max_of_e();
      if (me > kRescaleLog2) {
        resc = true;
        f = ex2_approx(-me);
        l_run *= f;
        m_run += me;
        shift(me);
      }
    }
    if (__any_sync(0xffffffffu, resc)) {
      tmem_wait_st();  // the first P has been written
      ls = exps();
    }
  }
  l_run += ls;
  if (__any_sync(0xffffffffu, resc)) {
    // (no later use of that region can have completed: the MMAs of step (t, g) wait for this warp)
    if (!mbar_wait(&bar.pv_done[C::sb(t, g - 1)], C::sp(t, g - 1))) return false;
    tc_fence_after();
#pragma unroll 1
    for (int c = 0; c < C::D; c += 32) {
      uint32_t o[32];
      tmem_ld32(o_addr + c, o);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
      tmem_st32(o_addr + c, o);
    }
  }
  tmem_wait_st();
  tc_fence_before();
  mbar_arrive(&bar.p_full[C::sb(t, g)]);
  return true;
}

// S_t = Q_t K^T for one key tile: D/16 MMAs (M128, N = BKV, K16) into TMEM
// column d; qdesc_t / kdesc_slot: shared-memory descriptors of Q_t and of the
// K ring slot (an operand at byte offset o is the descriptor plus o >> 4).
template <class C>
__device__ __forceinline__ void issue_s_mma(uint32_t d, uint64_t qdesc_t, uint64_t kdesc_slot) {
  constexpr uint32_t idesc_s = idesc_bf16_f32(128, C::BKV, false, false);
#pragma unroll
  for (int kk = 0; kk < C::D / 16; ++kk) {
    const uint64_t off_a = (uint64_t)(((kk >> 2) * C::CHUNK_Q + (kk & 3) * 32) >> 4);
    const uint64_t off_b = (uint64_t)(((kk >> 2) * C::CHUNK_KV + (kk & 3) * 32) >> 4);
    mma_bf16_ss(d, qdesc_t + off_a, kdesc_slot + off_b, idesc_s, kk != 0);
  }
}

// O_t (+)= P_t V for one key tile: BKV/16 MMAs (M128, N = D, K16), P_t from
// TMEM at column p (bf16 pairs over the S region), V MN-major from the ring
// slot; accumulate is false on an item's first key tile.
template <class C>
__device__ __forceinline__ void issue_pv_mma(uint32_t d, uint32_t p, uint64_t vdesc_slot, bool accumulate) {
  constexpr uint32_t idesc_o = idesc_bf16_f32(128, C::D, false, true);
#pragma unroll
  for (int kk = 0; kk < C::BKV / 16; ++kk)
    mma_bf16_ts(d, p + kk * 8, vdesc_slot + (uint64_t)((kk * 16 * 128) >> 4), idesc_o, accumulate || kk != 0);
}

// TMA loads of one K or V tile (D / 64 chunks of 64 columns) into a ring slot.
template <class C>
__device__ __forceinline__ void load_kv_tile(uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int col, int row) {
  mbar_expect_tx(bar, C::KV_BYTES);
  for (int c = 0; c < C::CH; ++c) tma_load_2d(dst + c * C::CHUNK_KV, map, bar, col + c * 64, row);
}

// Failure path (a wait ran out): the producer waits, bounded, until the last K
// and V loads of each ring have landed, so that no copy writes into the shared
// memory of a CTA that has left; the MMA thread waits, bounded, for the MMAs it
// has issued before tensor memory is freed.  Never called on the normal path.
template <class C>
__device__ __noinline__ void drain_loads(const AttnBars<C>& bar, int nk, int nv) {
  for (int j = nk > C::KVS ? nk - C::KVS : 0; j < nk; ++j) mbar_wait(&bar.k_full[C::slot(j)], C::round(j) & 1);
  for (int j = nv > C::KVS ? nv - C::KVS : 0; j < nv; ++j) mbar_wait(&bar.v_full[C::slot(j)], C::round(j) & 1);
}
__device__ __noinline__ void drain_mmas(uint64_t* drain) {
  mma_commit(drain);
  mbar_wait(drain, 0);
}

// The MMA warp's commits and operands.
template <class C>
struct AttnMma {
  const AttnBars<C>& bar;
  uint32_t tmem;
  uint64_t qdesc, kdesc, vdesc;
  __device__ __forceinline__ AttnMma(const AttnBars<C>& b, uint32_t tm, uint8_t* sQ, uint8_t* sK, uint8_t* sV)
      : bar(b), tmem(tm) {
    // Descriptors are built once; an operand at byte offset o from a base is
    // the base descriptor plus o >> 4 (the 14-bit address field cannot
    // overflow: shared memory ends below 256 KB).
    qdesc = smem_desc_sw128(smem_u32(sQ), 16, 1024);
    kdesc = smem_desc_sw128(smem_u32(sK), 16, 1024);
    vdesc = smem_desc_sw128(smem_u32(sV), C::CHUNK_KV, 1024);
  }
  // S_t = Q_t K^T of step g into its S region of tile t
  __device__ __forceinline__ void s_step(int t, int g) const {
    issue_s_mma<C>(tmem + C::sb(t, g) * C::BKV, qdesc + (uint64_t)((t * C::T_BYTES) >> 4),
                   kdesc + (uint64_t)((C::slot(g) * C::KV_BYTES) >> 4));
    mma_commit(&bar.s_full[C::sb(t, g)]);
    if (t == 1) mma_commit(&bar.k_empty[C::slot(g)]);
  }
  // O_t += P_t V of step g; accumulate is false on an item's first key tile
  __device__ __forceinline__ void pv_step(int t, int g, bool accumulate) const {
    issue_pv_mma<C>(tmem + C::o_col(t), tmem + C::sb(t, g) * C::BKV,
                    vdesc + (uint64_t)((C::slot(g) * C::KV_BYTES) >> 4), accumulate);
    mma_commit(&bar.pv_done[C::sb(t, g)]);
    if (t == 1) mma_commit(&bar.v_empty[C::slot(g)]);
  }
};

template <class C>
__global__ void __launch_bounds__(kAttnThreads, C::CTAS_PER_SM)
    attn_split_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                      const __grid_constant__ CUtensorMap tmV, AttnDev a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem + C::OFF_Q;
  uint8_t* sK = smem + C::OFF_K;
  uint8_t* sV = smem + C::OFF_V;
  const AttnBars<C> bar(smem + C::OFF_BAR);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int item = a.item_base + (int)blockIdx.x / a.splits, split = (int)blockIdx.x % a.splits;
  const int qt = item % a.nqp, h = item / a.nqp;
  const int nkv_all = (int)((a.nk + C::BKV - 1) / C::BKV);
  const int jb = (int)((int64_t)split * nkv_all / a.splits);  // this CTA's key tiles [jb, jb + nkv)
  const int nkv = (int)((int64_t)(split + 1) * nkv_all / a.splits) - jb;

  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
    bar.init();
  }
  if (warp == 1) tmem_alloc(bar.tmem_slot, C::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *bar.tmem_slot;
  pdl_wait();  // the set-up above overlaps the tail of the kernel before

  if (warp == 0) {
    if (lane == 0) {  // ---------------------------------------- TMA producer
      mbar_expect_tx(&bar.q_full[0], 2 * C::T_BYTES);
      for (int t = 0; t < 2; ++t)
        for (int c = 0; c < C::CH; ++c)
          tma_load_2d(sQ + t * C::T_BYTES + c * C::CHUNK_Q, &tmQ, &bar.q_full[0], a.q_col + h * C::D + c * 64,
                      qt * kBQ + t * kTileQ);
      int nk_issued = 0, nv_issued = 0;
      for (int j = 0; j < nkv; ++j) {
        const int st = C::slot(j);
        const uint32_t round = C::round(j);
        if (round > 0 && !mbar_wait(&bar.k_empty[st], (round - 1) & 1)) break;
        load_kv_tile<C>(sK + st * C::KV_BYTES, &tmK, &bar.k_full[st], a.k_col + h * C::D, (jb + j) * C::BKV);
        nk_issued = j + 1;
        if (round > 0 && !mbar_wait(&bar.v_empty[st], (round - 1) & 1)) break;
        load_kv_tile<C>(sV + st * C::KV_BYTES, &tmV, &bar.v_full[st], a.v_col + h * C::D, (jb + j) * C::BKV);
        nv_issued = j + 1;
      }
      if (nv_issued < nkv) {
        mbar_wait(&bar.q_full[0], 0);
        drain_loads<C>(bar, nk_issued, nv_issued);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------- MMA issuer
    // The whole warp walks the loop (descriptors and flags stay in uniform
    // registers) and one elected lane issues.
    const bool leader = elect_one();
    const AttnMma<C> mma(bar, tmem, sQ, sK, sV);
    bool ok = mbar_wait_warp(&bar.q_full[0], 0);
    auto issue_s = [&](int t, int j) -> bool {
      if (t == 0 && !mbar_wait_warp(&bar.k_full[C::slot(j)], C::round(j) & 1)) return false;
      tc_fence_after();
      if (leader) mma.s_step(t, j);
      __syncwarp();
      return true;
    };
    for (int n = 0; ok && n < 2 * nkv && n < C::NB; ++n) ok = issue_s(n & 1, n >> 1);
    for (int j = 0; ok && j < nkv; ++j) {
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        if (!mbar_wait_warp(&bar.p_full[C::sb(t, j)], C::sp(t, j))) { ok = false; break; }
        if (t == 0 && !mbar_wait_warp(&bar.v_full[C::slot(j)], C::round(j) & 1)) { ok = false; break; }
        tc_fence_after();
        if (leader) mma.pv_step(t, j, j != 0);
        __syncwarp();
        const int tn = (t + C::NB) & 1, jn = j + (t + C::NB) / 2;
        if (jn < nkv && !issue_s(tn, jn)) { ok = false; break; }
      }
    }
    if (!ok && leader) drain_mmas(bar.drain);
  } else {  // ---------------------------------------- softmax: warps 2-5 tile a, 6-9 tile b
    const int t = (warp - 2) >> 2;
    const int q = warp & 3;
    const int r = q * 32 + lane;  // row within the query tile == TMEM lane
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const uint32_t s_base = tmem + lane_base;
    const uint32_t o_addr = tmem + lane_base + C::o_col(t);
    float m_run = -INFINITY, l_run = 0.f;
    bool ok = true;
    // One key tile; the masked variant (keys past the end of the sequence)
    // is compiled separately and runs only on a partial last tile.
    auto step = [&](int j, auto masked) -> bool {
      return softmax_tile<C, decltype(masked)::value>(bar, t, j, j == 0, (int)(a.nk - (int64_t)(jb + j) * C::BKV),
                                                      s_base, o_addr, a.scale_log2, m_run, l_run);
    };
    const bool partial_last = (int64_t)(jb + nkv) * C::BKV > a.nk;
    for (int j = 0; j < nkv; ++j) {
      const bool ok_j = (j == nkv - 1 && partial_last) ? step(j, std::true_type{}) : step(j, std::false_type{});
      if (!ok_j) {
        ok = false;
        break;
      }
    }
    // ------------------------------ partial result of this key range: unnormalised O
    if (ok) ok = mbar_wait(&bar.pv_done[C::sb(t, nkv - 1)], C::sp(t, nkv - 1));
    tc_fence_after();
    const int64_t row = (int64_t)qt * kBQ + t * kTileQ + r;
    const int64_t slot = (int64_t)blockIdx.x * kBQ + t * kTileQ + r;
#pragma unroll 1
    for (int c = 0; c < C::D; c += 32) {
      uint32_t o[32];
      tmem_ld32(o_addr + c, o);
      tmem_wait_ld();
      if (!ok || row >= a.nq) continue;
      float* pp = a.part_o + slot * C::D + c;
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        *reinterpret_cast<float4*>(pp + i) = make_float4(__uint_as_float(o[i]), __uint_as_float(o[i + 1]),
                                                         __uint_as_float(o[i + 2]), __uint_as_float(o[i + 3]));
    }
    if (ok && row < a.nq) *reinterpret_cast<float2*>(a.part_ml + slot * 2) = make_float2(m_run, l_run);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, C::TMEM_COLS);
  }
}

// Whole items on persistent CTAs.  Each CTA walks the items
// item_base + blockIdx.x + k * gridDim.x; one counter g numbers its key-tile
// steps across items, and every per-step barrier phase and ring slot follows
// it.  Q_t of the next item is loaded once the current item's last S_t MMA
// has completed (q_empty), so the MMA warp issues the next item's first S
// right after the current item's last PV.  The output leaves through two
// staging boxes per softmax warp and TMA stores, which frees the softmax
// warps for the next item.
template <class C>
__global__ void __launch_bounds__(kAttnThreads, C::CTAS_PER_SM)
    attn_persist_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
                        AttnDev a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem + C::OFF_Q;
  uint8_t* sK = smem + C::OFF_K;
  uint8_t* sV = smem + C::OFF_V;
  const AttnBars<C> bar(smem + C::OFF_BAR_P);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int item0 = a.item_base + (int)blockIdx.x, item_step = (int)gridDim.x;
  const int n_items = item0 < a.item_end ? (a.item_end - 1 - item0) / item_step + 1 : 0;
  const int nkv = (int)((a.nk + C::BKV - 1) / C::BKV);
  const int total = n_items * nkv;  // key-tile steps of this CTA

  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
    tma_prefetch_desc(&tmO);
    bar.init();
  }
  if (warp == 1) tmem_alloc(bar.tmem_slot, C::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *bar.tmem_slot;
  pdl_wait();  // the set-up above overlaps the tail of the kernel before

  if (warp == 0) {
    if (lane == 0) {  // ---------------------------------------- TMA producer
      bool ok = true;
      int nk_issued = 0, nv_issued = 0;
      for (int k = 0, g = 0; ok && k < n_items; ++k) {
        const int item = item0 + k * item_step;
        const int qt = item % a.nqp, h = item / a.nqp;
        // Q_t of item k replaces Q_t of item k - 1 once that item's last S_t is
        // done; the item's first K goes out before Q_b, whose tile finishes later
        auto load_q = [&](int t) -> bool {
          if (k > 0 && !mbar_wait(&bar.q_empty[t], (k - 1) & 1)) return false;
          mbar_expect_tx(&bar.q_full[t], C::T_BYTES);
          for (int c = 0; c < C::CH; ++c)
            tma_load_2d(sQ + t * C::T_BYTES + c * C::CHUNK_Q, &tmQ, &bar.q_full[t], a.q_col + h * C::D + c * 64,
                        qt * kBQ + t * kTileQ);
          return true;
        };
        if (!load_q(0)) { ok = false; break; }
        for (int j = 0; ok && j < nkv; ++j, ++g) {
          const int st = C::slot(g);
          const uint32_t round = C::round(g);
          if (round > 0 && !mbar_wait(&bar.k_empty[st], (round - 1) & 1)) { ok = false; break; }
          load_kv_tile<C>(sK + st * C::KV_BYTES, &tmK, &bar.k_full[st], a.k_col + h * C::D, j * C::BKV);
          nk_issued = g + 1;
          if (j == 0 && !load_q(1)) { ok = false; break; }
          if (round > 0 && !mbar_wait(&bar.v_empty[st], (round - 1) & 1)) { ok = false; break; }
          load_kv_tile<C>(sV + st * C::KV_BYTES, &tmV, &bar.v_full[st], a.v_col + h * C::D, j * C::BKV);
          nv_issued = g + 1;
        }
      }
      // after a wait ran out: the last K and V loads of each ring have landed
      // (Q loads of an item are waited on by the MMA thread before any use)
      if (!ok) drain_loads<C>(bar, nk_issued, nv_issued);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------- MMA issuer
    // (whole warp walks, one elected lane issues, as in attn_split_kernel)
    const bool leader = elect_one();
    const AttnMma<C> mma(bar, tmem, sQ, sK, sV);
    // S_t of step g, which is key tile j of item k (jn, kn: of the next S to
    // issue); after an item's last key tile the producer may replace Q_t
    int jn = 0, kn = 0;
    auto issue_s = [&](int t, int g) -> bool {
      if (t == 0 && !mbar_wait_warp(&bar.k_full[C::slot(g)], C::round(g) & 1)) return false;
      if (jn == 0 && !mbar_wait_warp(&bar.q_full[t], kn & 1)) return false;
      tc_fence_after();
      if (leader) {
        mma.s_step(t, g);
        if (jn == nkv - 1) mma_commit(&bar.q_empty[t]);
      }
      __syncwarp();
      if (t == 1 && ++jn == nkv) {
        jn = 0;
        ++kn;
      }
      return true;
    };
    bool ok = true;
    for (int n = 0; ok && n < 2 * total && n < C::NB; ++n) ok = issue_s(n & 1, n >> 1);
    for (int g = 0, j = 0; ok && g < total; ++g) {
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        if (!mbar_wait_warp(&bar.p_full[C::sb(t, g)], C::sp(t, g))) { ok = false; break; }
        if (t == 0 && !mbar_wait_warp(&bar.v_full[C::slot(g)], C::round(g) & 1)) { ok = false; break; }
        tc_fence_after();
        if (leader) mma.pv_step(t, g, j != 0);
        __syncwarp();
        const int tn = (t + C::NB) & 1, gn = g + (t + C::NB) / 2;
        if (gn < total && !issue_s(tn, gn)) { ok = false; break; }
      }
      if (++j == nkv) j = 0;
    }
    if (!ok && leader) drain_mmas(bar.drain);
  } else {  // ---------------------------------------- softmax: warps 2-5 tile a, 6-9 tile b
    const int t = (warp - 2) >> 2;
    const int q = warp & 3;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const uint32_t s_base = tmem + lane_base;
    const uint32_t o_addr = tmem + lane_base + C::o_col(t);
    uint8_t* stage = smem + C::OFF_STAGE_P + (warp - 2) * 2 * C::STAGE_BOX;
    const int valid_last = (int)(a.nk - (int64_t)(nkv - 1) * C::BKV);  // keys of the last tile
    int n_st = 0;  // output boxes this warp has stored
    bool ok = true;
    for (int item = item0, g = 0; ok && item < a.item_end; item += item_step) {
      float m_run = -INFINITY, l_run = 0.f;
      for (int j = 0; j < nkv; ++j, ++g) {
        const bool ok_j = (j == nkv - 1 && valid_last < C::BKV)
                              ? softmax_tile<C, true>(bar, t, g, j == 0, valid_last, s_base, o_addr, a.scale_log2,
                                                      m_run, l_run)
                              : softmax_tile<C, false>(bar, t, g, j == 0, C::BKV, s_base, o_addr, a.scale_log2, m_run,
                                                       l_run);
        if (!ok_j) {
          ok = false;
          break;
        }
      }
      // ------------------------------------------------ output: O_t / l
      // (the next PV_t, which overwrites O_t, follows this warpgroup's next
      // p_full arrival, issued after these loads have completed)
      if (ok) ok = mbar_wait(&bar.pv_done[C::sb(t, g - 1)], C::sp(t, g - 1));
      ok = __all_sync(0xffffffffu, ok);  // the item loop continues for the whole warp or not at all
      tc_fence_after();
      const int qt = item % a.nqp, h = item / a.nqp;
      const int64_t row0 = (int64_t)qt * kBQ + t * kTileQ + q * 32;  // this warp's 32 rows
      const float inv = 1.0f / l_run;
#pragma unroll 1
      for (int c = 0; c < C::D; c += 32) {
        uint32_t o[32];
        tmem_ld32(o_addr + c, o);
        tmem_wait_ld();
        if (!ok || row0 >= a.nq) continue;  // warp-uniform
        // The warp's 32 x 32 box leaves through shared memory and one TMA
        // store (rows past nq are clipped by the tensor map).  Two boxes
        // alternate; the store issued two boxes ago must have read this one.
        uint8_t* box = stage + (n_st & 1) * C::STAGE_BOX;
        if (lane == 0 && n_st >= 2) bulk_wait_group_read<1>();
        __syncwarp();
        // row `lane`: 64 bytes as four 16-byte units, unit u stored at
        // u ^ ((lane >> 1) & 3) (the 64-byte swizzle: conflict-free writes)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint4 w;
          w.x = pack_bf16(__uint_as_float(o[8 * u + 0]) * inv, __uint_as_float(o[8 * u + 1]) * inv);
          w.y = pack_bf16(__uint_as_float(o[8 * u + 2]) * inv, __uint_as_float(o[8 * u + 3]) * inv);
          w.z = pack_bf16(__uint_as_float(o[8 * u + 4]) * inv, __uint_as_float(o[8 * u + 5]) * inv);
          w.w = pack_bf16(__uint_as_float(o[8 * u + 6]) * inv, __uint_as_float(o[8 * u + 7]) * inv);
          *reinterpret_cast<uint4*>(box + lane * 64 + ((u ^ ((lane >> 1) & 3)) << 4)) = w;
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          tma_store_2d(&tmO, box, a.o_col + h * C::D + c, (int)row0);
          bulk_commit_group();
        }
        ++n_st;
      }
    }
    if (lane == 0) bulk_wait_group<0>();  // output stores complete before the CTA ends
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, C::TMEM_COLS);
  }
}

// Merges the key-range parts of the split items: for every row,
// O = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s with M = max_s m_s.
// One warp per row (256 rows per item), D / 32 columns per lane.
template <int D>
__global__ void __launch_bounds__(256) attn_merge_kernel(AttnDev a, int item0, int tail, int splits) {
  pdl_wait();
  const int wrow = (int)(blockIdx.x * 8 + (threadIdx.x >> 5));  // row over all tail items
  const int lane = threadIdx.x & 31;
  if (wrow >= tail * kBQ) return;
  const int it = wrow / kBQ, rr = wrow % kBQ;
  const int item = item0 + it;
  const int qt = item % a.nqp, h = item / a.nqp;
  const int64_t row = (int64_t)qt * kBQ + rr;
  if (row >= a.nq) return;
  float M = -INFINITY;
  for (int sp = 0; sp < splits; ++sp) M = fmaxf(M, a.part_ml[((int64_t)(it * splits + sp) * kBQ + rr) * 2]);
  float acc[D / 32] = {};
  float L = 0.f;
  for (int sp = 0; sp < splits; ++sp) {
    const int64_t slot = (int64_t)(it * splits + sp) * kBQ + rr;
    const float w = ex2_approx(a.part_ml[slot * 2] - M);
    L += w * a.part_ml[slot * 2 + 1];
#pragma unroll
    for (int i = 0; i < D / 32; ++i) acc[i] = fmaf(w, a.part_o[slot * D + i * 32 + lane], acc[i]);
  }
  const float inv = 1.0f / L;
  if (!ACID_IN_BOUNDS(kSiteAttnMerge, row * a.ldo + a.o_col + h * D + D - 1, a.nq * a.ldo)) return;
  __nv_bfloat16* op = static_cast<__nv_bfloat16*>(a.out) + row * a.ldo + a.o_col + h * D;
#pragma unroll
  for (int i = 0; i < D / 32; ++i) op[i * 32 + lane] = __float2bfloat16_rn(acc[i] * inv);
}

template <class C>
acid_status launch_attn_tc(const AttnArgs& x, cudaStream_t s) {
  constexpr int D = C::D;
  static PerContext allowed, allowed_split;
  ACID_TRY(allow_smem(allowed, attn_persist_kernel<C>, C::SMEM_P));
  CUtensorMap tq, tk, tv;
  ACID_TRY(make_tmap_bf16(&tq, x.q, x.nq, x.ldq, x.ldq, kTileQ));
  ACID_TRY(make_tmap_bf16(&tk, x.k, x.nk, x.ldk, x.ldk, C::BKV));
  ACID_TRY(make_tmap_bf16(&tv, x.v, x.nk, x.ldv, x.ldv, C::BKV));
  AttnDev a;
  a.nq = x.nq;
  a.nk = x.nk;
  a.q_col = x.q_col;
  a.k_col = x.k_col;
  a.v_col = x.v_col;
  a.out = x.out;
  a.ldo = x.ldo;
  a.o_col = x.o_col;
  a.scale_log2 = (float)(1.4426950408889634 / sqrt((double)D));
  a.nqp = (int)((x.nq + kBQ - 1) / kBQ);
  a.item_base = 0;
  a.item_end = 0;
  a.splits = 1;
  a.part_o = nullptr;
  a.part_ml = nullptr;
  const int items = a.nqp * x.heads;
  const int nkv_all = (int)((x.nk + C::BKV - 1) / C::BKV);
  // Items fill whole waves of persistent CTAs, CTAS_PER_SM on an SM (measured at
  // head dim 128, us, persistent / one item per CTA: 4846 tokens, 24 heads 179 /
  // 188; 7800, 12 heads 248 / 254; 1100, 12 heads 18.5 / 22.2).  Long key ranges:
  // the items of a last, partial wave are split along the key range so that
  // they fill one wave together, and their partial results are merged.  Short
  // key ranges: the persistent CTAs take all items, and the few CTAs that take
  // one item more cost less than a split wave's start-up and merge (measured:
  // 109 against 121 us for 32760 x 512 keys).
  const int slots = num_sms() * C::CTAS_PER_SM;
  const int full = (items / slots) * slots, tail = items - full;
  int splits = tail > 0 ? std::min(std::min(kAttnPartCtas, slots) / tail, nkv_all) : 1;
  const size_t part_need = (size_t)tail * splits * kBQ * (D + 2) * sizeof(float);
  const bool short_keys = x.nk <= 8 * D;
  const bool split_tail =
      !short_keys && full > 0 && tail > 0 && splits >= 2 && x.part != nullptr && x.part_bytes >= part_need;
  ProfScope prof(PROF_ATTENTION, 4.0 * (double)x.nq * (double)x.nk * D * x.heads, s);
  const int main_items = split_tail ? full : items;
  // output: 32-row x 32-column boxes, one per softmax warp and column chunk
  CUtensorMap to;
  ACID_TRY(make_tmap_bf16_box(&to, x.out, x.nq, x.ldo, x.ldo, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B));
  a.item_end = main_items;
  if constexpr (C::CTAS_PER_SM == 1) {
    if (split_tail) ACID_TRY(allow_smem(allowed_split, attn_split_kernel<C>, C::SMEM));
  }
  launch_pdl(attn_persist_kernel<C>, std::min(main_items, slots), kAttnThreads, C::SMEM_P, s, tq, tk, tv, to, a);
  ACID_CHECK_LAUNCH();
  if (!split_tail) return ACID_OK;
  a.item_base = full;
  a.splits = splits;
  a.part_o = static_cast<float*>(x.part);
  a.part_ml = a.part_o + (size_t)tail * splits * kBQ * D;
  if constexpr (C::CTAS_PER_SM == 1) {
    launch_pdl(attn_split_kernel<C>, tail * splits, kAttnThreads, C::SMEM, s, tq, tk, tv, a);
    ACID_CHECK_LAUNCH();
    launch_pdl(attn_merge_kernel<D>, tail * kBQ / 8, 256, 0, s, a, full, tail, splits);
    ACID_CHECK_LAUNCH();
  }
  return ACID_OK;
}

// ---------------------------------------------------------------- fp32 path
// Tiled flash attention on the FP32 pipes.  A CTA takes BQ query rows of one
// head; its four groups of four warps walk the key range in interleaved tiles
// of 32 keys, each group with its own K and V buffers, running max and
// partial output, and the groups' parts are merged through shared memory at
// the end.  The group split is what fills the SMs when there are few query
// tiles (256 tokens x 4 heads are 64 tiles of 16 rows) and gives each SM 16
// warps to hide the loads behind.
//   A half-warp owns QT = BQ / 8 query rows: lane kg of it computes the scores
// of keys kg and kg + 16 with those rows (16-byte shared loads along the head
// dim; the K rows are padded by 16 bytes, so 16 rows cover all banks), the row
// max goes through half-warp shuffles, P through shared memory, and the same
// lanes then accumulate QT rows x D / 16 columns of the output.  The row sum
// stays per lane until the end.  K(j + 1) loads (cp.async) while P V runs and
// V(j) while the scores of tile j are formed.
//   Measured at 256 tokens, 4 heads of 64: 10.2 us, against 161.7 us for one
// warp per query row (a serial loop over the keys with a shuffle tree and two
// exponentials per key).  What bounds it there is the latency of two key tiles
// per group (about 4 us of FP32 work) plus load, merge and launch.
constexpr int kF32Groups = 4, kF32Keys = 32;

template <int D, int BQ>
struct AttnF32Cfg {
  static constexpr int QT = BQ / 8;    // query rows per half-warp
  static constexpr int LDK = D + 4;    // padded K (and Q) row, floats
  static constexpr int LDP = kF32Keys + 4;
  static constexpr int K_FLOATS = kF32Keys * LDK, V_FLOATS = kF32Keys * D;
  static constexpr int OFF_Q = 0;
  static constexpr int OFF_P = BQ * LDK;                           // [group][BQ][LDP]
  static constexpr int OFF_KV = OFF_P + kF32Groups * BQ * LDP;     // [group][K | V]; reused for the merge
  static constexpr int FLOATS = OFF_KV + kF32Groups * (K_FLOATS + V_FLOATS);
  static constexpr int SMEM = FLOATS * 4;
  static_assert(kF32Groups * BQ * (D + 2) <= kF32Groups * (K_FLOATS + V_FLOATS), "merge buffers fit the K/V area");
  static_assert(SMEM <= 227 * 1024, "fp32 attention shared memory");
};

struct AttnF32Args {
  const float* q;
  const float* k;
  const float* v;
  float* out;
  int64_t ldq, ldk, ldv, ldo, nq, nk;
  float scale;
  int vec;  // 1: rows of q, k and v are 16-byte aligned
};

// ROWS rows of D floats (row stride ld in global memory, lds in shared
// memory) by `threads` threads; rows from `valid_rows` on are zero.
template <int D, int ROWS>
__device__ __forceinline__ void load_rows_f32(float* dst, int lds, const float* src, int64_t ld, int64_t valid_rows,
                                              int tid, int threads, int vec) {
  if (vec) {
    for (int i = tid; i < ROWS * (D / 4); i += threads) {
      const int r = i / (D / 4), c = (i % (D / 4)) * 4;
      const bool ok = r < valid_rows;
      cp_async<16>(dst + r * lds + c, src + (ok ? (int64_t)r * ld + c : 0), ok);
    }
  } else {
    for (int i = tid; i < ROWS * D; i += threads) {
      const int r = i / D, c = i % D;
      const bool ok = r < valid_rows;
      cp_async<4>(dst + r * lds + c, src + (ok ? (int64_t)r * ld + c : 0), ok);
    }
  }
}

template <int D, int BQ>
__global__ void __launch_bounds__(128 * kF32Groups) attn_f32_kernel(AttnF32Args a) {
  pdl_wait();
  using C = AttnF32Cfg<D, BQ>;
  constexpr int QT = C::QT, KT = kF32Keys / 16, NC = D / 32;  // NC column pairs per lane
  extern __shared__ __align__(16) float fsm[];
  const int g = threadIdx.x >> 7, t = threadIdx.x & 127;  // group, thread in the group
  const int hw = t >> 4, kg = t & 15;                     // half-warp (rows hw * QT ..), lane in it
  const int64_t q0 = (int64_t)blockIdx.x * BQ;
  const int h = blockIdx.y;
  float* sq = fsm + C::OFF_Q;
  float* sp = fsm + C::OFF_P + g * BQ * C::LDP + hw * QT * C::LDP;
  float* sk = fsm + C::OFF_KV + g * (C::K_FLOATS + C::V_FLOATS);
  float* sv = sk + C::K_FLOATS;
  const float* kh = a.k + h * D;
  const float* vh = a.v + h * D;
  const int ntiles = (int)((a.nk + kF32Keys - 1) / kF32Keys);
  auto load_k = [&](int j) {
    const int64_t k0 = (int64_t)j * kF32Keys;
    load_rows_f32<D, kF32Keys>(sk, C::LDK, kh + k0 * a.ldk, a.ldk, a.nk - k0, t, 128, a.vec);
  };
  auto load_v = [&](int j) {
    const int64_t k0 = (int64_t)j * kF32Keys;
    load_rows_f32<D, kF32Keys>(sv, D, vh + k0 * a.ldv, a.ldv, a.nk - k0, t, 128, a.vec);
  };
  // Q rows (all groups), this group's first K and V tiles: one commit group each
  load_rows_f32<D, BQ>(sq, C::LDK, a.q + q0 * a.ldq + h * D, a.ldq, a.nq - q0, threadIdx.x, blockDim.x, a.vec);
  if (g < ntiles) load_k(g);
  cp_async_commit();
  if (g < ntiles) load_v(g);
  cp_async_commit();
  cp_async_wait<1>();
  __syncthreads();  // Q and every group's first K tile

  float o[QT][2 * NC] = {};
  float m[QT], l[QT];
#pragma unroll
  for (int i = 0; i < QT; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
  }
  const float* qrow = sq + hw * QT * C::LDK;
  for (int j = g; j < ntiles; j += kF32Groups) {
    // Scores of QT rows x KT keys, summed in pairs, quads, blocks of 16 and then
    // over the blocks.  One chain over the head dim takes up to 4% less time, but
    // had 1.5 times the error of a lane-wise tree at few keys (16 tokens: 2.0e-7
    // of the output against 1.3e-7; this order 1.2e-7; 2048 tokens 5.0e-7 against
    // 1.1e-6; this order 4.3e-7).
    float s[QT][KT] = {};
#pragma unroll 1
    for (int d0 = 0; d0 < D; d0 += 16) {
      float u[QT][KT];
#pragma unroll
      for (int d = 0; d < 16; d += 4) {
        float4 qv[QT], kv[KT];
#pragma unroll
        for (int i = 0; i < QT; ++i) qv[i] = *reinterpret_cast<const float4*>(qrow + i * C::LDK + d0 + d);
#pragma unroll
        for (int c = 0; c < KT; ++c) kv[c] = *reinterpret_cast<const float4*>(sk + (kg + 16 * c) * C::LDK + d0 + d);
#pragma unroll
        for (int i = 0; i < QT; ++i)
#pragma unroll
          for (int c = 0; c < KT; ++c) {
            const float x = fmaf(qv[i].y, kv[c].y, qv[i].x * kv[c].x) + fmaf(qv[i].w, kv[c].w, qv[i].z * kv[c].z);
            u[i][c] = d == 0 ? x : u[i][c] + x;
          }
      }
#pragma unroll
      for (int i = 0; i < QT; ++i)
#pragma unroll
        for (int c = 0; c < KT; ++c) s[i][c] += u[i][c];
    }
    group_sync(1 + g, 128);  // every warp of the group has read the K tile
    if (j + kF32Groups < ntiles) load_k(j + kF32Groups);
    cp_async_commit();
    const int64_t left = a.nk - (int64_t)j * kF32Keys;  // keys of this tile
#pragma unroll
    for (int i = 0; i < QT; ++i) {
      float mt = -INFINITY;
#pragma unroll
      for (int c = 0; c < KT; ++c) {
        s[i][c] = kg + 16 * c < left ? s[i][c] * a.scale : -INFINITY;
        mt = fmaxf(mt, s[i][c]);
      }
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, off));
      const float mn = fmaxf(m[i], mt);
      const float ref = mn == -INFINITY ? 0.f : mn;  // no finite score yet: every term below is 0
      const float corr = expf(m[i] - ref);
      m[i] = mn;
      l[i] *= corr;
#pragma unroll
      for (int c = 0; c < 2 * NC; ++c) o[i][c] *= corr;
#pragma unroll
      for (int c = 0; c < KT; ++c) {
        const float p = kg + 16 * c < left ? expf(s[i][c] - ref) : 0.f;
        l[i] += p;
        sp[i * C::LDP + kg + 16 * c] = p;
      }
    }
    cp_async_wait<1>();      // V(j) has landed (this thread's copies)
    group_sync(1 + g, 128);  // ... and every thread's; P is written
    const int kmax = left < kF32Keys ? (int)left : kF32Keys;
#pragma unroll 2
    for (int k = 0; k < kmax; k += 4) {  // V rows past the end are zero, and so is P
      float4 pv[QT];
#pragma unroll
      for (int i = 0; i < QT; ++i) pv[i] = *reinterpret_cast<const float4*>(sp + i * C::LDP + k);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        float2 vv[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) vv[c] = *reinterpret_cast<const float2*>(sv + (k + kk) * D + 32 * c + 2 * kg);
#pragma unroll
        for (int i = 0; i < QT; ++i) {
          const float p = kk == 0 ? pv[i].x : kk == 1 ? pv[i].y : kk == 2 ? pv[i].z : pv[i].w;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            o[i][2 * c] = fmaf(p, vv[c].x, o[i][2 * c]);
            o[i][2 * c + 1] = fmaf(p, vv[c].y, o[i][2 * c + 1]);
          }
        }
      }
    }
    cp_async_wait<0>();      // K(j + groups) has landed
    group_sync(1 + g, 128);  // V and P have been read
    if (j + kF32Groups < ntiles) load_v(j + kF32Groups);
    cp_async_commit();
  }
  cp_async_wait<0>();
  // ---- merge: [group][BQ][D] partial outputs, then [group][BQ] {m, l}
#pragma unroll
  for (int i = 0; i < QT; ++i)
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);
  __syncthreads();  // every group has finished with its K and V buffers
  float* mo = fsm + C::OFF_KV;
  float2* ml = reinterpret_cast<float2*>(mo + kF32Groups * BQ * D);
#pragma unroll
  for (int i = 0; i < QT; ++i) {
    const int r = hw * QT + i;
#pragma unroll
    for (int c = 0; c < NC; ++c)
      *reinterpret_cast<float2*>(mo + (g * BQ + r) * D + 32 * c + 2 * kg) = make_float2(o[i][2 * c], o[i][2 * c + 1]);
    if (kg == 0) ml[g * BQ + r] = make_float2(m[i], l[i]);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < BQ * D; i += blockDim.x) {
    const int r = i / D, c = i % D;
    if (q0 + r >= a.nq) break;
    float mx = -INFINITY;
#pragma unroll
    for (int gg = 0; gg < kF32Groups; ++gg) mx = fmaxf(mx, ml[gg * BQ + r].x);
    float acc = 0.f, den = 0.f;
#pragma unroll
    for (int gg = 0; gg < kF32Groups; ++gg) {
      const float2 e = ml[gg * BQ + r];
      if (gg >= ntiles) break;  // a group without a tile holds no part
      const float w = expf(e.x - mx);
      den = fmaf(w, e.y, den);
      acc = fmaf(w, mo[(gg * BQ + r) * D + c], acc);
    }
    const int64_t at = (q0 + r) * a.ldo + h * D + c;
    if (!ACID_IN_BOUNDS(kSiteAttnF32, at, a.nq * a.ldo)) continue;
    a.out[at] = acc / den;
  }
}

template <int D, int BQ>
acid_status attn_f32_launch(const AttnF32Args& a, int heads, cudaStream_t s) {
  using C = AttnF32Cfg<D, BQ>;
  static PerContext allowed;
  ACID_TRY(allow_smem(allowed, attn_f32_kernel<D, BQ>, C::SMEM));
  const dim3 grid((unsigned)((a.nq + BQ - 1) / BQ), (unsigned)heads);
  launch_pdl(attn_f32_kernel<D, BQ>, grid, 128 * kF32Groups, C::SMEM, s, a);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

template <int D>
acid_status launch_attn_f32(const AttnArgs& x, cudaStream_t s) {
  AttnF32Args a;
  a.q = static_cast<const float*>(x.q) + x.q_col;
  a.k = static_cast<const float*>(x.k) + x.k_col;
  a.v = static_cast<const float*>(x.v) + x.v_col;
  a.out = static_cast<float*>(x.out) + x.o_col;
  a.ldq = x.ldq;
  a.ldk = x.ldk;
  a.ldv = x.ldv;
  a.ldo = x.ldo;
  a.nq = x.nq;
  a.nk = x.nk;
  a.scale = (float)(1.0 / sqrt((double)D));
  a.vec = aligned(a.q, 16) && aligned(a.k, 16) && aligned(a.v, 16) && x.ldq % 4 == 0 && x.ldk % 4 == 0 &&
          x.ldv % 4 == 0;
  // 32-row tiles reuse each K and V value for twice the rows; 16-row tiles
  // while the 32-row ones would leave SMs without a CTA
  if ((x.nq + 31) / 32 * x.heads < num_sms()) return attn_f32_launch<D, 16>(a, x.heads, s);
  return attn_f32_launch<D, 32>(a, x.heads, s);
}

}  // namespace

acid_status attention_forward(int dtype, const AttnArgs& x, cudaStream_t s) {
  ACID_REQUIRE(x.nk > 0 && x.nq >= 0 && x.heads > 0, ACID_ERR_INVALID_ARG, "attention: bad shape");
  if (x.nq == 0) return ACID_OK;  // no query rows: nothing is read, pointers may be null
  ACID_REQUIRE(x.q && x.k && x.v && x.out, ACID_ERR_INVALID_ARG, "attention: null pointer");
  if (dtype == ACID_FP32) {
    ACID_REQUIRE(x.head_dim % 32 == 0 && x.head_dim <= 128, ACID_ERR_UNSUPPORTED,
                 "attention fp32: head_dim must be 32, 64, 96 or 128");
    switch (x.head_dim) {
      case 32: return launch_attn_f32<32>(x, s);
      case 64: return launch_attn_f32<64>(x, s);
      case 96: return launch_attn_f32<96>(x, s);
      default: return launch_attn_f32<128>(x, s);
    }
  }
  ACID_REQUIRE(x.head_dim == 64 || x.head_dim == 128, ACID_ERR_UNSUPPORTED, "attention bf16: head_dim must be 64 or 128");
  ACID_REQUIRE(x.q_col % 8 == 0 && x.k_col % 8 == 0 && x.v_col % 8 == 0 && x.o_col % 8 == 0 && x.ldo % 8 == 0,
               ACID_ERR_UNSUPPORTED, "attention bf16: column offsets must be multiples of 8");
  ACID_REQUIRE(aligned(x.out, 16), ACID_ERR_UNSUPPORTED, "attention bf16: output must be 16-byte aligned");
  if (x.head_dim == 128) return launch_attn_tc<AttnCfg<128, 128>>(x, s);
  // Measured at head dim 64 (us, 64-key / 128-key tiles), 17776 x 226 keys, 30
  // heads: 45.0 / 53.6; 4726 x 400: 21.4 / 24.5; x 450: 23.7 / 24.5; x 512: 23.2 /
  // 22.6; self-attention of 500 tokens 9.6 / 8.2, of 4726 tokens (64-key tiles,
  // two CTAs on an SM, as every range took them once) 177 / 147.
  if (x.nk <= 448) return launch_attn_tc<AttnCfg<64, 64>>(x, s);
  return launch_attn_tc<AttnCfg<64, 128>>(x, s);
}

ACID_DEVICE_FLAG_READER(take_device_error_attention)
ACID_BOUNDS_READER(take_bounds_attention)

}  // namespace acid
