// Linear layers of the DiT block.
//
// bf16: a persistent tcgen05 GEMM.  A pair of CTAs on two SMs
// (tcgen05.mma.cta_group::2) computes 256 x bn output tiles with the fp32
// accumulator in tensor memory (TMEM), double-buffered.  Warp 0 streams the A
// and B tiles with TMA (128-byte swizzle) through an mbarrier ring; warp 1
// issues tcgen05.mma; warps 2-9 read the accumulator back with tcgen05.ld (one
// thread per output row) and apply the fused epilogue (bias, GELU-tanh, 3D
// RoPE of q/k, gated or plain residual) before a TMA store.  A dual-stream
// layer's text and video rows, with weights of their own, share a launch.
// Long-K GEMMs inside a block can finish their last round as split-K units
// (see splitk_plan).
//
// fp32: a register-tiled SIMT GEMM with the same epilogue (the fp32 mode's
// 1e-4 tolerance rules out tf32 tensor cores).
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "internal.h"

namespace acid {

namespace {

// Epilogue parameters as passed to the kernels.
struct EpiDev {
  int kind;
  const float* bias;
  const float* bias_t;  // bias of the text rows' problem (dual-stream launches)
  const float* gate_v;
  const float* gate_t;
  int64_t gate_split;
  const void* res;
  int64_t ldr;
  int res_fp32;
  int64_t row_base;
  RopeTable rope;
  int64_t rope_first_video;
  int d, head_dim;
};

EpiDev to_dev(const Epilogue& e) {
  EpiDev d;
  d.kind = e.kind;
  d.bias = e.bias;
  d.bias_t = e.text_bias;
  d.gate_v = e.gate_video;
  d.gate_t = e.gate_text ? e.gate_text : e.gate_video;
  d.gate_split = e.gate_split;
  d.res = e.residual;
  d.ldr = e.ldr;
  d.res_fp32 = e.res_fp32 ? 1 : 0;
  d.row_base = e.row_base;
  d.rope = e.rope;
  d.rope_first_video = e.rope_first_video;
  d.d = e.d;
  d.head_dim = e.head_dim;
  return d;
}

// Video position -> (frame, row, column) of the latent grid in 32-bit
// arithmetic.  Positions are below 2^24 (checked on the host), so the float
// quotient n * (1/d) is within one of floor(n / d) and one correction step
// makes it exact.
struct RopePos {
  int f, h, w;
};
__device__ __forceinline__ int div_small(int n, int d, float inv_d) {
  int q = (int)((float)n * inv_d);
  const int r = n - q * d;
  q += (r >= d) - (r < 0);
  return q;
}
__device__ __forceinline__ RopePos rope_pos(const RopeTable& t, int pos) {
  const int hw = t.grid_h * t.grid_w;
  RopePos p;
  p.f = div_small(pos, hw, t.inv_hw);
  const int rem = pos - p.f * hw;
  p.h = div_small(rem, t.grid_w, t.inv_w);
  p.w = rem - p.h * t.grid_w;
  return p;
}

// Table entry (cos, sin) of the RoPE angle of pair `jj` (within the head) at a
// decomposed position.
__device__ __forceinline__ const float2& rope_cs(const RopeTable& t, const RopePos& p, int jj) {
  if (jj < t.pairs_t) return t.table[p.f * t.pairs_t + jj];
  jj -= t.pairs_t;
  const int off_h = t.grid_f * t.pairs_t;
  if (jj < t.pairs_h) return t.table[off_h + p.h * t.pairs_h + jj];
  jj -= t.pairs_h;
  const int off_w = off_h + t.grid_h * t.pairs_h;
  return t.table[off_w + p.w * t.pairs_w + jj];
}
// (debug builds) the table entry's index lies inside the table
__device__ __forceinline__ bool rope_in_bounds(const RopeTable& t, const float2& e) {
  const int64_t n = (int64_t)t.grid_f * t.pairs_t + (int64_t)t.grid_h * t.pairs_h + (int64_t)t.grid_w * t.pairs_w;
  return ACID_IN_BOUNDS(kSiteGemmRope, &e - t.table, n);
}

// The (cos, sin) of the 16 consecutive pairs from j0 on (within the head) at a
// position.  The table index is formed with selects, so that the 16 loads go
// out together: behind a branch per pair each waited for the one before.
__device__ __forceinline__ void rope_cs16(const RopeTable& t, const RopePos& p, int j0, float2* cs) {
  const int end_t = t.pairs_t, end_h = end_t + t.pairs_h;
  const int off_h = t.grid_f * t.pairs_t, off_w = off_h + t.grid_h * t.pairs_h;
  const int base_t = p.f * t.pairs_t;
  const int base_h = off_h + p.h * t.pairs_h - end_t, base_w = off_w + p.w * t.pairs_w - end_h;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int jj = j0 + k;
    const float2* e = t.table + (jj + (jj < end_t ? base_t : jj < end_h ? base_h : base_w));
    cs[k] = rope_in_bounds(t, *e) ? __ldg(e) : make_float2(1.f, 0.f);
  }
}

// Applies the epilogue to the adjacent outputs (grow, col) and (grow, col+1).
// r0/r1: residual values (read by the caller) for the residual kinds.
template <bool kFastGelu>
__device__ __forceinline__ void epi_pair(const EpiDev& e, int64_t grow, int col, float& a, float& b, float r0,
                                         float r1) {
  if (e.bias) {
    a += e.bias[col];
    b += e.bias[col + 1];
  }
  switch (e.kind) {
    case EPI_GELU:
      a = gelu_tanh<kFastGelu>(a);
      b = gelu_tanh<kFastGelu>(b);
      break;
    case EPI_ROPE_QKV:
      if (col < 2 * e.d && grow >= e.rope_first_video) {
        const float2 cs = rope_cs(e.rope, rope_pos(e.rope, (int)(grow - e.rope_first_video)), (col % e.head_dim) >> 1);
        const float x0 = a, x1 = b;
        a = x0 * cs.x - x1 * cs.y;
        b = x0 * cs.y + x1 * cs.x;
      }
      break;
    case EPI_GATED_RES: {
      const float* g = grow < e.gate_split ? e.gate_t : e.gate_v;
      a = fmaf(g[col], a, r0);
      b = fmaf(g[col + 1], b, r1);
      break;
    }
    case EPI_RES:
      a += r0;
      b += r1;
      break;
    default:
      break;
  }
}

__host__ __device__ __forceinline__ bool epi_reads_res(int kind) { return kind == EPI_GATED_RES || kind == EPI_RES; }

constexpr int BM = 128, BK = 64;  // rows of A per CTA, depth of a k-step
constexpr int kEpiWarps = 8;
constexpr int kGemmThreads = 64 + 32 * kEpiWarps;

struct GemmDims {
  int64_t M;
  int N, K;
  // split-K launches only: work unit = (tile, split); split s covers k-blocks
  // [s kb_split, (s + 1) kb_split) and stores its raw fp32 accumulator at
  // rows s m_pad + row of the partial buffer
  int splits = 1, kb_split = 0;
  int64_t m_pad = 0;
  // output columns per tile (a multiple of 32, at most 256) and the depth of
  // the operand ring
  int bn = 256, stages = 6;
  // dual-stream launches: rows [0, l_text) are multiplied with the text
  // weights, in mt_text row tiles of their own; 0: one problem
  int l_text = 0, mt_text = 0;
  // residual rows that overlap (row stride below N, as in a row repeated for
  // every output row): not expressible as a tensor map, read with plain loads
  int res_direct = 0;
};

// GELU (tanh form) of a packed pair, with the arithmetic of gelu_tanh<true>
// done two lanes at a time: u = sqrt(2/pi) (x + 0.044715 x^3), out = h + h tanh(u)
// with h = x / 2.
__device__ __forceinline__ uint64_t gelu_x2(uint64_t x) {
  const uint64_t c3 = f2_pack(0.044715f, 0.044715f), k0 = f2_pack(0.7978845608028654f, 0.7978845608028654f);
  const uint64_t half = f2_pack(0.5f, 0.5f);
  const uint64_t u = f2_mul(k0, f2_fma(f2_mul(c3, x), f2_mul(x, x), x));
  float u0, u1;
  f2_unpack(u, u0, u1);
  const uint64_t t = f2_pack(tanh_fast(u0), tanh_fast(u1));
  const uint64_t h = f2_mul(half, x);
  return f2_fma(h, t, h);
}

// Kinds whose epilogue reads no residual.
template <int KIND>
constexpr bool kNoResidual = !(KIND == EPI_GATED_RES || KIND == EPI_RES);

// Bias of a chunk's 32 columns, the same for every lane (broadcast loads
// through the read-only path; 16-byte loads where the vector is aligned).
__device__ __forceinline__ void load_bias32(const float* src, int col0, float* bias) {
  if (src == nullptr) {
#pragma unroll
    for (int k = 0; k < 32; ++k) bias[k] = 0.f;
  } else if ((reinterpret_cast<uintptr_t>(src + col0) & 15) == 0) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(src + col0) + k);
      bias[4 * k] = t.x; bias[4 * k + 1] = t.y; bias[4 * k + 2] = t.z; bias[4 * k + 3] = t.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 32; ++k) bias[k] = __ldg(src + col0 + k);
  }
}

// Epilogue of one 32-row x 32-column chunk of a kind without a residual, in
// the layout tcgen05.ld delivers (thread = row, 32 consecutive columns): the
// bias and the kind's arithmetic in registers, then the output box written
// once into the warp's stage in the tensor store's swizzled layout (fp32:
// 128-byte rows, 16-byte unit u of row r at u ^ (r & 7); bf16: 64-byte rows,
// unit u at u ^ ((r >> 1) & 3); both place the 32 rows' units of a given u in
// distinct bank groups) and handed to one TMA store, which clips rows past M.
// Shared-memory traffic is one write and one TMA read of the box.  The caller
// makes sure the store that last read this stage has finished reading.
template <int KIND, bool O32>
__device__ __forceinline__ void epilogue_rows(const CUtensorMap* tmO, uint8_t* stage, int64_t store_row0, int col0,
                                              const uint32_t* r, const float* bias, const float2* cs) {
  const int lane = threadIdx.x & 31;
  uint64_t v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k)
    v[k] = f2_add(f2_pack(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1])),
                  f2_pack(bias[2 * k], bias[2 * k + 1]));
  if constexpr (KIND == EPI_GELU) {
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = gelu_x2(v[k]);
  } else if constexpr (KIND == EPI_ROPE_QKV) {
    if (cs != nullptr) {
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        float x0, x1;
        f2_unpack(v[k], x0, x1);
        v[k] = f2_pack(x0 * cs[k].x - x1 * cs[k].y, x0 * cs[k].y + x1 * cs[k].x);
      }
    }
  }
  if constexpr (O32) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      float a0, a1, a2, a3;
      f2_unpack(v[2 * u], a0, a1);
      f2_unpack(v[2 * u + 1], a2, a3);
      *reinterpret_cast<float4*>(stage + lane * 128 + ((u ^ (lane & 7)) << 4)) = make_float4(a0, a1, a2, a3);
    }
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      uint32_t w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float a0, a1;
        f2_unpack(v[4 * u + q], a0, a1);
        w[q] = pack_bf16(a0, a1);
      }
      *reinterpret_cast<uint4*>(stage + lane * 64 + ((u ^ ((lane >> 1) & 3)) << 4)) =
          make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  fence_proxy_async_smem();
  __syncwarp();
  if (lane == 0) {
    tma_store_2d(tmO, stage, col0, (int)store_row0);
    bulk_commit_group();
  }
}

// One chunk of a kind without a residual: accumulator and bias loads, the
// stage (bf16 output: two 2 KB stages per warp used in turn, so a chunk waits
// only for the store before last; fp32 output: one 4 KB stage), epilogue_rows.
template <int KIND, bool O32>
__device__ __forceinline__ void tma_kind_chunk(const GemmDims& g, const EpiDev& e, const CUtensorMap* tmO,
                                               uint8_t* stage, uint32_t taddr, int64_t row0, int64_t store_row0,
                                               int col0, const float* bias_src, bool live, int& nstore) {
  const int lane = threadIdx.x & 31;
  uint32_t r[32];
  float bias[32];
  tmem_ld32(taddr, r);
  if (live) load_bias32(bias_src, col0, bias);
  // RoPE of q and k on video rows: the chunk's 16 pairs lie in one head
  // (head_dim is a power of two >= 32); other rows are rotated by (1, 0)
  float2 cs[KIND == EPI_ROPE_QKV ? 16 : 1];
  bool rotate = false;
  if constexpr (KIND == EPI_ROPE_QKV) {
    rotate = live && col0 < 2 * e.d;  // warp-uniform
    if (rotate) {
      const int64_t row = row0 + lane, grow = row + e.row_base;
      const bool video = grow >= e.rope_first_video && row < g.M;
      const RopePos pos = rope_pos(e.rope, video ? (int)(grow - e.rope_first_video) : 0);
      rope_cs16(e.rope, pos, (col0 & (e.head_dim - 1)) >> 1, cs);
      if (!video) {
#pragma unroll
        for (int k = 0; k < 16; ++k) cs[k] = make_float2(1.f, 0.f);
      }
    }
  }
  tmem_wait_ld();
  if (!live) return;
  uint8_t* st = stage;
  if constexpr (O32) {
    if (lane == 0) bulk_wait_group_read<0>();
  } else {
    st += (nstore & 1) * 2048;
    if (lane == 0) bulk_wait_group_read<1>();
  }
  __syncwarp();
  epilogue_rows<KIND, O32>(tmO, st, store_row0, col0, r, bias, rotate ? cs : nullptr);
  ++nstore;
}

// One chunk of a residual kind of the pair kernel, also in the accumulator's
// layout.  The residual box (32 x 32, TMA-loaded into the warp's box `box` in
// the swizzled layouts of epilogue_rows) is read by the lane that owns the
// row, the result is written back over it and leaves by TMA store; two boxes
// alternate.  Accumulator, bias and gate loads are issued before the wait for
// the box: loaded after it, group by group, the gates alone cost 1500 of
// 4100 SM clocks per chunk.  next(): issues the residual load of the chunk after this
// one into the other box, once the store that last used it has read it.
// Returns false if the wait ran out.
template <int KIND, bool R32, bool O32, typename Next>
__device__ __forceinline__ bool res_kind_chunk(const GemmDims& g, const EpiDev& e, const CUtensorMap* tmO, uint8_t* box,
                                               uint64_t* box_full, uint32_t phase, uint32_t taddr, int64_t row0,
                                               int col0, const float* bias_src, Next next) {
  const int lane = threadIdx.x & 31;
  uint32_t r[32];
  float bv[32], gv[32];
  tmem_ld32(taddr, r);
  load_bias32(bias_src, col0, bv);
  if constexpr (KIND == EPI_GATED_RES)
    load_bias32(row0 + lane + e.row_base < e.gate_split ? e.gate_t : e.gate_v, col0, gv);
  const bool ok = g.res_direct || mbar_wait_warp(box_full, phase);
  tmem_wait_ld();
  if (!ok) return false;
  uint64_t v[16];
#pragma unroll
  for (int u = 0; u < 4; ++u) {  // 8 columns of this lane's residual row
    float rv[8] = {};
    if (g.res_direct) {
      const int64_t at = (row0 + lane) * e.ldr + col0 + 8 * u;
      if (row0 + lane < g.M && ACID_IN_BOUNDS(kSiteGemmResidual, at + 7, (g.M - 1) * e.ldr + g.N)) {
        if constexpr (R32)
          load8(static_cast<const float*>(e.res) + at, rv);
        else
          load8(static_cast<const __nv_bfloat16*>(e.res) + at, rv);
      }
    } else if constexpr (R32) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 t = *reinterpret_cast<const float4*>(box + lane * 128 + (((2 * u + h) ^ (lane & 7)) << 4));
        rv[4 * h] = t.x; rv[4 * h + 1] = t.y; rv[4 * h + 2] = t.z; rv[4 * h + 3] = t.w;
      }
    } else {
      load8(reinterpret_cast<const __nv_bfloat16*>(box + lane * 64 + ((u ^ ((lane >> 1) & 3)) << 4)), rv);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = 8 * u + 2 * k;
      const uint64_t acc = f2_add(f2_pack(__uint_as_float(r[c]), __uint_as_float(r[c + 1])), f2_pack(bv[c], bv[c + 1]));
      const uint64_t rr = f2_pack(rv[2 * k], rv[2 * k + 1]);
      if constexpr (KIND == EPI_GATED_RES)
        v[4 * u + k] = f2_fma(f2_pack(gv[c], gv[c + 1]), acc, rr);
      else
        v[4 * u + k] = f2_add(acc, rr);
    }
  }
  next();
  __syncwarp();  // every lane has read its residual row
  if constexpr (O32) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      float a0, a1, a2, a3;
      f2_unpack(v[2 * u], a0, a1);
      f2_unpack(v[2 * u + 1], a2, a3);
      *reinterpret_cast<float4*>(box + lane * 128 + ((u ^ (lane & 7)) << 4)) = make_float4(a0, a1, a2, a3);
    }
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      uint32_t w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float a0, a1;
        f2_unpack(v[4 * u + q], a0, a1);
        w[q] = pack_bf16(a0, a1);
      }
      *reinterpret_cast<uint4*>(box + lane * 64 + ((u ^ ((lane >> 1) & 3)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  fence_proxy_async_smem();
  __syncwarp();
  if (lane == 0) {
    tma_store_2d(tmO, box, col0, (int)row0);
    bulk_commit_group();
  }
  return true;
}

// ===========================================================================
// tcgen05 GEMM on SM pairs (cta_group::2), persistent
//
// A cluster of two CTAs on two SMs computes 256 x bn output tiles (bn up to
// 256, see pick_bn): each CTA stages its own 128 rows of A and its own bn / 2
// rows of B per 64-wide k-step, and one thread of CTA rank 0 issues M256 N(bn)
// K16 MMAs that read both CTAs' shared memory and write each CTA's 128 x bn
// fp32 accumulator into that CTA's TMEM.  At bn = 256 this moves 32 KB per SM
// and k-step into shared memory for 128 x 256 x 64 MACs, against 48 KB for a
// single-SM 128 x 256 tile.  Tiles go N fastest, so the pairs running together
// share A row blocks in L2 and the weight tiles stay L2-resident; the TMEM
// accumulator is double-buffered, so the epilogue of tile i overlaps the MMAs
// of tile i + 1.
//   warp 0   TMA producer in both CTAs; both CTAs' loads count on rank 0's
//            full[s] barrier (rank 0 expects the bytes of both);
//   warp 1   rank 0: MMA issuer; each k-step is committed to empty[s] of both
//            CTAs, each tile to acc_full[b] of both CTAs;
//   warps 2-9 epilogue of this CTA's 128 accumulator rows; one lane per warp
//            then arrives on rank 0's acc_empty[b], which counts the epilogue
//            warps of both CTAs.
//   What bounds it: long mainloops run into the power cap (FFN1 at 32760 rows,
// 1536 -> 8960 with GELU: 529 to 545 us on several GPUs, 1650 to 1705 TFLOP/s, at
// 1.42 to 1.48 GHz, and 477 us in runs of 20 ms; 579 to 590 us before the issue
// loops below kept to uniform registers).  A k-step's floor is the
// issue of its loads and MMAs: 240 SM clocks at bn = 32, where it was 580.
// ===========================================================================
struct Tc2Cfg {
  static constexpr int MAX_BN = 256;           // output columns per pair tile (g.bn: a multiple of 32)
  static constexpr int A_BYTES = BM * BK * 2;  // this CTA's 128 rows of A; its bn / 2 rows of B follow
  static constexpr int MAX_STAGES = 12;
  // Operand ring and epilogue boxes share shared memory: kinds without a
  // residual have six 32 KB stages and 4 KB per epilogue warp, residual kinds
  // five stages and two 4 KB boxes per warp.
  static constexpr int RING = 6 * 32768, RING_RES = 5 * 32768;
  static constexpr int WARP = 4096, WARP_RES = 8192;
  static constexpr int SMEM = RING + kEpiWarps * WARP + 1024 + 512;
  __host__ __device__ static constexpr int stage_bytes(int bn) { return A_BYTES + bn * BK; }
  static int stages(int bn, bool res) { return std::min(MAX_STAGES, (res ? RING_RES : RING) / stage_bytes(bn)); }
  static constexpr uint32_t TMEM_COLS = 2 * MAX_BN;  // double-buffered 128 x bn accumulator
};
static_assert(Tc2Cfg::SMEM <= 232448, "pair GEMM shared memory");
static_assert(Tc2Cfg::RING_RES + kEpiWarps * Tc2Cfg::WARP_RES == Tc2Cfg::RING + kEpiWarps * Tc2Cfg::WARP,
              "one shared memory size for both layouts");

// Where a pair tile lies: its first row, its first column and whose rows it
// holds (dual-stream launches: the text rows' tiles come first).
struct TilePos {
  int row, col;
  bool text;
};
__device__ __forceinline__ TilePos tile_pos(const GemmDims& g, int tile, int num_n) {
  const int m = tile / num_n;
  TilePos t;
  t.text = m < g.mt_text;
  t.row = t.text ? m * 2 * BM : g.l_text + (m - g.mt_text) * 2 * BM;
  t.col = (tile - m * num_n) * g.bn;
  return t;
}

template <int KIND, bool R32, bool O32, bool SPLIT = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
    gemm_tc2_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmR,
                    const __grid_constant__ CUtensorMap tmBt, const __grid_constant__ CUtensorMap tmOt, GemmDims g,
                    EpiDev e) {
  using C = Tc2Cfg;
  constexpr bool RES = !kNoResidual<KIND>;
  constexpr int RING = RES ? C::RING_RES : C::RING, WARP = RES ? C::WARP_RES : C::WARP;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + RING + kEpiWarps * WARP);
  uint64_t* full = bars;                       // [MAX_STAGES]
  uint64_t* empty = full + C::MAX_STAGES;      // [MAX_STAGES]
  uint64_t* acc_full = empty + C::MAX_STAGES;  // [2]
  uint64_t* acc_empty = acc_full + 2;          // [2] (rank 0's counts both CTAs' epilogue warps)
  uint64_t* drain = acc_empty + 2;             // failure path: the MMAs issued so far have completed
  uint64_t* res_full = drain + 1;              // [epilogue warp][2] residual box loaded
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(res_full + 2 * kEpiWarps);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = (int)blockIdx.x >> 1, npairs = (int)gridDim.x >> 1;
  const int num_kb = SPLIT ? g.kb_split : (g.K + BK - 1) / BK;
  const int num_n = (g.N + g.bn - 1) / g.bn;
  const int num_m = g.mt_text + (int)((g.M - g.l_text + 2 * BM - 1) / (2 * BM));
  const int num_units = SPLIT ? num_m * num_n * g.splits : num_m * num_n;  // (tile, split) pairs
  const int stages = g.stages, stage_bytes = C::stage_bytes(g.bn);

  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 2 * kEpiWarps);
    }
    if constexpr (RES)
      for (int i = 0; i < 2 * kEpiWarps; ++i) mbar_init(&res_full[i], 1);
    mbar_init(drain, 1);
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, C::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist before any cross-CTA arrival
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();  // the set-up above overlaps the tail of the kernel before

  if (warp == 0) {
    // TMA producer (both CTAs): one continuous stage ring across tiles; the
    // whole warp walks the loop and one elected lane issues, as for the MMAs
    const bool leader = elect_one();
    const uint32_t full0 = mapa_shared(smem_u32(full), 0);  // rank 0's full[0]
    int s = 0, issued = 0;
    uint32_t ph = 1;  // parity of the previous use of the stage (a fresh barrier passes on 1)
    bool ok = true;
    for (int unit = pair; ok && unit < num_units; unit += npairs) {
      const TilePos t = tile_pos(g, SPLIT ? unit / g.splits : unit, num_n);
      const int k0 = SPLIT ? (unit % g.splits) * num_kb * BK : 0;
      const CUtensorMap* tb = t.text ? &tmBt : &tmB;
      const int arow = t.row + (int)rank * BM, brow = t.col + (int)rank * (g.bn / 2);
      for (int kb = 0; kb < num_kb; ++kb) {
        if (!mbar_wait_warp(&empty[s], ph)) { ok = false; break; }
        if (leader) {
          if (rank == 0) mbar_expect_tx(&full[s], 2 * stage_bytes);
          uint8_t* st = smem + s * stage_bytes;
          tma_load_2d_pair(st, &tmA, full0 + 8 * s, k0 + kb * BK, arow);
          tma_load_2d_pair(st + C::A_BYTES, tb, full0 + 8 * s, k0 + kb * BK, brow);
        }
        __syncwarp();
        ++issued;
        if (++s == stages) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    // After a wait ran out: rank 0 waits (bounded) for the last `stages`
    // stages it expected to land.  Rank 1's loads count on rank 0's
    // barriers, which rank 1 cannot poll; it idles about 2^16 clocks, far
    // above the latency of a 32 KB load, before both CTAs meet at the exit.
    if (!ok && leader) {
      if (rank == 0) {
        for (int j = std::max(0, issued - stages); j < issued; ++j) mbar_wait(&full[j % stages], (j / stages) & 1);
      } else {
        const long long t0 = clock64();
        while (clock64() - t0 < (1LL << 16)) {
        }
      }
    }
  } else if (warp == 1) {
    // MMA issuer (rank 0 only).  The whole warp walks the loop, so that the
    // descriptors stay in uniform registers, and one elected lane issues:
    // with the loop in a single-lane branch a k-step's four MMAs took 257 SM
    // clocks to issue and a whole k-step 530, above the 512 they run for.
    if (rank == 0) {
      const bool leader = elect_one();
      const uint32_t idesc = idesc_bf16_f32(2 * BM, g.bn, false, false);
      const uint32_t empty_l = smem_u32(empty), accf_l = smem_u32(acc_full);
      const uint64_t adesc = smem_desc_sw128(smem_u32(smem), 16, 1024);
      const uint64_t bdesc = smem_desc_sw128(smem_u32(smem + C::A_BYTES), 16, 1024);
      int s = 0, local = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int unit = pair; ok && unit < num_units; unit += npairs, ++local) {
        const int b = local & 1, use = local >> 1;
        if (use > 0 && !__all_sync(0xffffffffu, mbar_wait_cluster(&acc_empty[b], (use - 1) & 1))) { ok = false; break; }
        tc_fence_after();
        const uint32_t d = tmem + b * C::MAX_BN;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!mbar_wait_warp(&full[s], ph)) { ok = false; break; }
          tc_fence_after();
          const uint64_t off = (uint64_t)((s * stage_bytes) >> 4);
          if (leader) {
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              mma_bf16_ss_pair(d, adesc + off + 2 * k, bdesc + off + 2 * k, idesc, (kb | k) != 0);
            mma_commit_both(empty_l + 8 * s);
          }
          __syncwarp();
          if (++s == stages) {
            s = 0;
            ph ^= 1;
          }
        }
        if (ok && leader) mma_commit_both(accf_l + 8 * b);
        __syncwarp();
      }
      if (!ok && leader) {
        mma_commit_pair(smem_u32(drain));
        mbar_wait(drain, 0);
      }
    }
  } else {  // epilogue: warps 2..9 of each CTA, this CTA's 128 rows of the pair tile
    // lane quarter = warp % 4; the tile's 32-column chunks alternate between
    // the two warps of a quarter
    const int q = warp & 3, half = (warp - 2) >> 2;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    uint8_t* stage = smem + RING + (warp - 2) * WARP;
    const uint32_t acc_empty0 = mapa_shared(smem_u32(acc_empty), 0);
    const int row_in = (int)rank * BM + q * 32, nch = g.bn / 32;
    uint64_t* rfull = res_full + 2 * (warp - 2);
    // Residual kinds: the position (unit, chunk) of the next residual load;
    // seek() moves it on to the first chunk from there with rows and columns
    // to store.  Loads are numbered like the chunks that consume them.
    int lu = pair, lc = half, lrow = 0, lcol = 0, loads = 0, nchunk = 0;
    auto seek = [&]() {
      for (; lu < num_units; lu += npairs, lc = half) {
        const TilePos t = tile_pos(g, lu, num_n);
        lrow = t.row + row_in;
        lcol = t.col + 32 * lc;
        if (lc < nch && lcol < g.N && lrow < (t.text ? g.l_text : (int)g.M)) return true;
      }
      return false;
    };
    auto load_next = [&]() {  // lane 0
      if (!seek()) return;
      uint64_t* bar = &rfull[loads & 1];
      mbar_expect_tx(bar, R32 ? 4096 : 2048);
      tma_load_2d(stage + (loads & 1) * 4096, &tmR, bar, lcol, lrow);
      ++loads;
      lc += 2;
    };
    if constexpr (RES) {
      if (lane == 0 && !g.res_direct) {
        load_next();
        load_next();
      }
    }
    int local = 0, nstore = 0;
    for (int unit = pair; unit < num_units; unit += npairs, ++local) {
      const int b = local & 1, use = local >> 1;
      const TilePos t = tile_pos(g, SPLIT ? unit / g.splits : unit, num_n);
      const int64_t row0 = t.row + row_in;
      const bool rows_live = row0 < (t.text ? (int64_t)g.l_text : g.M);
      const CUtensorMap* to = t.text ? &tmOt : &tmO;
      const float* bias = t.text ? e.bias_t : e.bias;
      bool ok = mbar_wait(&acc_full[b], use & 1);
      tc_fence_after();
#pragma unroll 1
      for (int c = half; c < nch; c += 2) {
        const uint32_t taddr = tmem + lane_base + b * C::MAX_BN + 32 * c;
        const int col0 = t.col + 32 * c;
        const bool live = ok && rows_live && col0 < g.N;  // warp-uniform
        if constexpr (!RES) {
          const int64_t store_row0 = SPLIT ? row0 + (int64_t)(unit % g.splits) * g.m_pad : row0;
          tma_kind_chunk<KIND, O32>(g, e, to, stage, taddr, row0, store_row0, col0, bias, live, nstore);
        } else if (live) {
          const int x = nchunk & 1;
          auto next = [&]() {  // the other box: its chunk's store was issued one chunk ago
            if (lane == 0 && nchunk > 0) {
              bulk_wait_group_read<0>();
              if (!g.res_direct) load_next();
            }
          };
          ok = res_kind_chunk<KIND, R32, O32>(g, e, to, stage + x * 4096, &rfull[x], (nchunk >> 1) & 1, taddr, row0,
                                              col0, bias, next);
          if (!ok) break;
          ++nchunk;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acc_empty0 + 8 * b);
      if (!ok) break;
    }
    if (lane == 0) {
      // after a wait ran out: the residual loads already issued land before the CTA exits
      if constexpr (RES)
        for (; nchunk < loads; ++nchunk) mbar_wait(&rfull[nchunk & 1], (nchunk >> 1) & 1);
      bulk_wait_group<0>();  // tensor stores complete before the CTA exits
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // no CTA leaves while its peer may still signal its barriers
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, C::TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------
// TMA descriptor encoding through the driver entry point (no -lcuda needed)
// ---------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

}  // namespace

// Row-major matrix [rows, cols] of 2-byte (bf16) or 4-byte (fp32) elements
// with row stride ld (elements), boxes of box_rows x box_cols, the given
// swizzle, zero fill out of bounds (loads) and clipping (stores).
acid_status make_tmap_2d(CUtensorMap* map, CUtensorMapDataType type, int esize, const void* base, int64_t rows,
                         int64_t cols, int64_t ld, int box_cols, int box_rows, CUtensorMapSwizzle swizzle) {
  auto fn = encode_fn();
  ACID_REQUIRE(fn != nullptr, ACID_ERR_CUDA, "cuTensorMapEncodeTiled entry point unavailable");
  ACID_REQUIRE(aligned(base, 16) && (ld * esize) % 16 == 0, ACID_ERR_UNSUPPORTED,
               "TMA operand must be 16-byte aligned with a row stride that is a multiple of 16 bytes");
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * esize)};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1u, 1u};
  CUresult r = fn(map, type, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  ACID_REQUIRE(r == CUDA_SUCCESS, ACID_ERR_CUDA, "cuTensorMapEncodeTiled failed (code " + std::to_string((int)r) + ")");
  return ACID_OK;
}

acid_status make_tmap_bf16_box(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld,
                               int box_cols, int box_rows, CUtensorMapSwizzle swizzle) {
  return make_tmap_2d(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, rows, cols, ld, box_cols, box_rows, swizzle);
}

// Boxes of box_rows x 64 columns with 128-byte swizzle (the MMA operand layout).
acid_status make_tmap_bf16(CUtensorMap* map, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  return make_tmap_bf16_box(map, base, rows, cols, ld, 64, box_rows, CU_TENSOR_MAP_SWIZZLE_128B);
}

namespace {

// The GEMM output as the epilogue's tensor stores see it: 32 x 32 boxes, the
// swizzle of the box layout in epilogue_rows (128-byte rows for fp32,
// 64-byte rows for bf16).
acid_status make_tmap_out(CUtensorMap* map, void* out, int64_t M, int N, int64_t ldo, bool fp32) {
  return fp32 ? make_tmap_2d(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, out, M, N, ldo, 32, 32,
                             CU_TENSOR_MAP_SWIZZLE_128B)
              : make_tmap_2d(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, out, M, N, ldo, 32, 32,
                             CU_TENSOR_MAP_SWIZZLE_64B);
}

// An instance of the pair kernel and its count of CTA pairs that can be
// resident at once (clusters are placed within a GPC, so this can be below half
// the SM count), always positive on success.
using PairKernel = decltype(&gemm_tc2_kernel<EPI_BIAS, false, false>);
struct PairInstance {
  PairKernel kernel;
  acid_status (*pairs)(int* n);
};

template <int KIND, bool R32, bool O32, bool SPLIT>
acid_status max_pairs(int* pairs) {
  static PerContext known;
  return known.get(pairs, [](int* n) {
    const PairKernel kernel = gemm_tc2_kernel<KIND, R32, O32, SPLIT>;
    // the dynamic shared memory limit must be raised before the query (and the launch)
    ACID_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Tc2Cfg::SMEM));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * 76, 1, 1);
    cfg.blockDim = dim3(kGemmThreads, 1, 1);
    cfg.dynamicSmemBytes = Tc2Cfg::SMEM;
    ACID_CUDA(cudaOccupancyMaxActiveClusters(n, kernel, &cfg));
    ACID_REQUIRE(*n > 0, ACID_ERR_CUDA, "linear: no resident CTA pair for the pair GEMM");
    return ACID_OK;
  });
}

template <int KIND, bool R32, bool O32, bool SPLIT = false>
PairInstance pair_instance() {
  return {gemm_tc2_kernel<KIND, R32, O32, SPLIT>, max_pairs<KIND, R32, O32, SPLIT>};
}

// The instance that applies an epilogue.
template <int KIND, bool R32 = false>
PairInstance pair_instance_out(const Epilogue& e) {
  return e.out_fp32 ? pair_instance<KIND, R32, true>() : pair_instance<KIND, R32, false>();
}
PairInstance pair_instance_for(const Epilogue& e) {
  switch (e.kind) {
    case EPI_GELU: return pair_instance_out<EPI_GELU>(e);
    case EPI_ROPE_QKV: return pair_instance_out<EPI_ROPE_QKV>(e);
    case EPI_GATED_RES:
      return e.res_fp32 ? pair_instance_out<EPI_GATED_RES, true>(e) : pair_instance_out<EPI_GATED_RES>(e);
    case EPI_RES: return e.res_fp32 ? pair_instance_out<EPI_RES, true>(e) : pair_instance_out<EPI_RES>(e);
    default: return pair_instance_out<EPI_BIAS>(e);
  }
}

int64_t pair_row_tiles(int64_t M, int64_t text_rows) {
  return (text_rows + 2 * BM - 1) / (2 * BM) + (M - text_rows + 2 * BM - 1) / (2 * BM);
}

// Output columns per tile: the width with the lowest estimated time, in SM
// clocks, of the pair that gets the most tiles.  A k-step runs for 2 bn clocks
// on the tensor cores plus about 75, and not below its issue cost; each tile
// adds about 500 and the last tile's epilogue 700 per pair of 32-column
// chunks.  Narrower tiles win where a last round of 256-wide ones leaves pairs
// idle.  Measured at 256 columns and at the width chosen (us a call, back to back
// over inputs that change, in runs too short for the power cap; calls below 10 us
// are bound by the calling program): 7797 x 1920 x 1920 (M x K x N) gated residual
// 43.6, 39.3 at 160 (41.7 at 128, 42.3 at 192); 7800 x 1536 x 4608 66.7, 65.4 at
// 192; 512 x 1536 x 3072 13.2, 9.3 at 96; 64 x 8960 x 1536 45.6, 22.9 at 32; the
// widest layer of a 480p step stays at 256 (1536 -> 8960: 477 against 481 at 224).
int pick_bn(int64_t m_tiles, int N, int K, int pairs) {
  const int64_t num_kb = (K + BK - 1) / BK;
  int best = Tc2Cfg::MAX_BN;
  int64_t best_cost = INT64_MAX;
  for (int bn = Tc2Cfg::MAX_BN; bn >= 32; bn -= 32) {
    const int64_t tiles = m_tiles * ((N + bn - 1) / bn), rounds = (tiles + pairs - 1) / pairs;
    const int64_t step = std::max(2 * bn + 75, 220 + bn / 2);
    const int64_t cost = rounds * (num_kb * step + 500) + 700 * ((bn + 63) / 64);
    if (cost < best_cost) {
      best = bn;
      best_cost = cost;
    }
  }
  return best;
}

// Tensor maps of one launch of the pair kernel.
struct PairMaps {
  CUtensorMap a, b, o, r, bt, ot;
};

acid_status launch_pairs(PairKernel kernel, const PairMaps& t, const GemmDims& g, const Epilogue& epi, int64_t units,
                         int pairs, cudaStream_t s) {
  const int grid = 2 * (int)std::min<int64_t>(units, pairs);
  launch_pdl(kernel, grid, kGemmThreads, Tc2Cfg::SMEM, s, t.a, t.b, t.o, t.r, t.bt, t.ot, g, to_dev(epi));
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

acid_status launch_tc2(const void* A, int64_t lda, int64_t M, int K, const void* W, int N, void* out, int64_t ldo,
                       const Epilogue& epi, cudaStream_t s) {
  const PairInstance inst = pair_instance_for(epi);
  int pairs = 0;
  ACID_TRY(inst.pairs(&pairs));
  const int64_t m_tiles = pair_row_tiles(M, epi.text_rows);
  const int bn = pick_bn(m_tiles, N, K, pairs);
  const bool res = epi_reads_res(epi.kind);
  PairMaps t;
  ACID_TRY(make_tmap_bf16(&t.a, A, M, K, lda, BM));
  ACID_TRY(make_tmap_bf16(&t.b, W, N, K, K, bn / 2));
  ACID_TRY(make_tmap_out(&t.o, out, M, N, ldo, epi.out_fp32));
  t.r = t.o;
  const bool res_direct = res && epi.ldr < N;
  if (res && !res_direct)
    ACID_TRY(make_tmap_out(&t.r, const_cast<void*>(epi.residual), M, N, epi.ldr, epi.res_fp32));
  t.bt = t.b;
  t.ot = t.o;
  GemmDims g{M, N, K};
  g.bn = bn;
  g.stages = Tc2Cfg::stages(bn, res);
  g.res_direct = res_direct;
  if (epi.text_rows > 0) {  // the output map of the text rows ends with them
    ACID_TRY(make_tmap_bf16(&t.bt, epi.text_w, N, K, K, bn / 2));
    ACID_TRY(make_tmap_out(&t.ot, out, epi.text_rows, N, ldo, epi.out_fp32));
    g.l_text = (int)epi.text_rows;
    g.mt_text = (int)((epi.text_rows + 2 * BM - 1) / (2 * BM));
  }
  const int64_t tiles = m_tiles * ((N + bn - 1) / bn);
  ProfScope prof(PROF_LINEAR, 2.0 * (double)M * N * K, s);
  return launch_pairs(inst.kernel, t, g, epi, tiles, pairs, s);
}

// ---------------------------------------------------------------------------
// Split-K last round of the pair GEMM.  With K long, a persistent launch
// whose last round keeps only a few CTA pairs busy spends a whole tile's
// mainloop on it.  The rows that fill whole rounds then run as usual, and
// the remaining rows run as (tile, k-split) units, one per pair, each storing
// its raw fp32 accumulator into scratch; splitk_fixup_kernel adds a row's
// partials in split order and applies the epilogue.
struct SplitKPlan {
  int64_t rows_main = 0;  // rows of the ordinary launch (whole 256-row tiles)
  int splits = 0, kb_split = 0;
  int64_t m_pad = 0;      // tail rows rounded up to 256 (per-split stride of the scratch)
};

bool splitk_plan(int64_t M, int N, int K, size_t ws_bytes, int pairs, SplitKPlan* p) {
  constexpr int64_t bm = 2 * BM;
  const int64_t n_tiles = (N + Tc2Cfg::MAX_BN - 1) / Tc2Cfg::MAX_BN, m_tiles = (M + bm - 1) / bm;
  const int64_t tiles = m_tiles * n_tiles, num_kb = (K + BK - 1) / BK;
  if (num_kb < 64) return false;  // short mainloops: the last round is cheap
  const int64_t full = tiles / pairs, last = tiles - full * pairs;
  if (full < 1 || last == 0 || 2 * last >= pairs) return false;
  const int64_t rows_main = (full * pairs / n_tiles) * bm;
  if (rows_main <= 0 || rows_main >= M) return false;
  const int64_t tail = M - rows_main, tail_tiles = ((tail + bm - 1) / bm) * n_tiles;
  const int64_t splits = std::min<int64_t>({pairs / tail_tiles, num_kb / 16, 16});
  if (splits < 3) return false;
  p->rows_main = rows_main;
  p->splits = (int)splits;
  p->kb_split = (int)((num_kb + splits - 1) / splits);
  p->m_pad = ((tail + bm - 1) / bm) * bm;
  return (size_t)splits * p->m_pad * N * sizeof(float) <= ws_bytes;
}

template <int KIND, bool R32, bool O32>
__global__ void __launch_bounds__(256) splitk_fixup_kernel(const float* __restrict__ part, int splits, int64_t m_pad,
                                                           int64_t M, int N, void* out, int64_t ldo, EpiDev e) {
  pdl_wait();
  const int64_t npair = N / 2, total = M * npair;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
    const int64_t row = i / npair;
    const int col = (int)(i - row * npair) * 2;
    float a = 0.f, b = 0.f;
    for (int sp = 0; sp < splits; ++sp) {
      const float2 v = *reinterpret_cast<const float2*>(part + ((int64_t)sp * m_pad + row) * N + col);
      a += v.x;
      b += v.y;
    }
    float r0 = 0.f, r1 = 0.f;
    if constexpr (KIND == EPI_GATED_RES || KIND == EPI_RES) {
      if constexpr (R32) {
        const float2 rv = *reinterpret_cast<const float2*>(static_cast<const float*>(e.res) + row * e.ldr + col);
        r0 = rv.x;
        r1 = rv.y;
      } else {
        const __nv_bfloat16* res = static_cast<const __nv_bfloat16*>(e.res) + row * e.ldr + col;
        const uint32_t rv = *reinterpret_cast<const uint32_t*>(res);
        r0 = bf16_lo(rv);
        r1 = bf16_hi(rv);
      }
    }
    epi_pair<true>(e, row + e.row_base, col, a, b, r0, r1);
    if (!ACID_IN_BOUNDS(kSiteGemmStore, row * ldo + col + 1, (M - 1) * ldo + N)) continue;
    if constexpr (O32)
      *reinterpret_cast<float2*>(static_cast<float*>(out) + row * ldo + col) = make_float2(a, b);
    else
      *reinterpret_cast<uint32_t*>(static_cast<__nv_bfloat16*>(out) + row * ldo + col) = pack_bf16(a, b);
  }
}

template <int KIND, bool R32, bool O32>
acid_status launch_splitk_fixup(const SplitKPlan& sp, const float* part, int64_t M, int N, void* out, int64_t ldo,
                                const Epilogue& epi, cudaStream_t s) {
  const int64_t total = M * (N / 2);
  const int grid = (int)std::min<int64_t>((total + 255) / 256, (int64_t)num_sms() * 8);
  launch_pdl(splitk_fixup_kernel<KIND, R32, O32>, grid, 256, 0, s, part, sp.splits, sp.m_pad, M, N, out, ldo,
             to_dev(epi));
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

template <int KIND, bool R32 = false>
acid_status launch_splitk_fixup_kind(const SplitKPlan& sp, const float* part, int64_t M, int N, void* out,
                                     int64_t ldo, const Epilogue& epi, cudaStream_t s) {
  return epi.out_fp32 ? launch_splitk_fixup<KIND, R32, true>(sp, part, M, N, out, ldo, epi, s)
                      : launch_splitk_fixup<KIND, R32, false>(sp, part, M, N, out, ldo, epi, s);
}

// The split-K units of the tail rows [M rows of A], then the fixup into out.
acid_status launch_tc2_splitk(const void* A, int64_t lda, int64_t M, int K, const void* W, int N, void* out,
                              int64_t ldo, const Epilogue& epi, const SplitKPlan& sp, cudaStream_t s) {
  const PairInstance inst = pair_instance<EPI_BIAS, false, true, true>();
  int pairs = 0;
  ACID_TRY(inst.pairs(&pairs));
  float* part = static_cast<float*>(epi.splitk_ws);
  PairMaps t;
  ACID_TRY(make_tmap_bf16(&t.a, A, M, K, lda, BM));
  ACID_TRY(make_tmap_bf16(&t.b, W, N, K, K, Tc2Cfg::MAX_BN / 2));
  ACID_TRY(make_tmap_out(&t.o, part, (int64_t)sp.splits * sp.m_pad, N, N, true));
  t.r = t.ot = t.o;
  t.bt = t.b;
  GemmDims g{M, N, K};  // 256 columns per tile
  g.splits = sp.splits;
  g.kb_split = sp.kb_split;
  g.m_pad = sp.m_pad;
  Epilogue raw;  // the accumulator as it is: no bias, fp32
  raw.out_fp32 = true;
  const int64_t units = ((M + 2 * BM - 1) / (2 * BM)) * ((N + Tc2Cfg::MAX_BN - 1) / Tc2Cfg::MAX_BN) * sp.splits;
  {
    ProfScope prof(PROF_LINEAR, 2.0 * (double)M * N * K, s);
    ACID_TRY(launch_pairs(inst.kernel, t, g, raw, units, pairs, s));
  }
  switch (epi.kind) {
    case EPI_GELU: return launch_splitk_fixup_kind<EPI_GELU>(sp, part, M, N, out, ldo, epi, s);
    case EPI_ROPE_QKV: return launch_splitk_fixup_kind<EPI_ROPE_QKV>(sp, part, M, N, out, ldo, epi, s);
    case EPI_GATED_RES:
      return epi.res_fp32 ? launch_splitk_fixup_kind<EPI_GATED_RES, true>(sp, part, M, N, out, ldo, epi, s)
                          : launch_splitk_fixup_kind<EPI_GATED_RES, false>(sp, part, M, N, out, ldo, epi, s);
    case EPI_RES:
      return epi.res_fp32 ? launch_splitk_fixup_kind<EPI_RES, true>(sp, part, M, N, out, ldo, epi, s)
                          : launch_splitk_fixup_kind<EPI_RES, false>(sp, part, M, N, out, ldo, epi, s);
    default: return launch_splitk_fixup_kind<EPI_BIAS>(sp, part, M, N, out, ldo, epi, s);
  }
}

// ===========================================================================
// fp32 SIMT GEMM
//
// A CTA computes a TM x TN output tile with four groups of 64 threads that
// take the 32-deep K slices in turn (group g: slices g, g + 4, ...), each with
// its own three-stage cp.async ring, and adds the groups' accumulators in
// group order in shared memory before the epilogue.  Splitting K inside the
// CTA keeps eight warps busy on a tile as small as 16 x 32, so a layer of a
// few hundred rows (the fp32 models' size) still spreads over the SMs.  A
// thread holds TM / 8 x TN / 8 outputs: rows 2 ty + {0, 1} + 16 i and columns
// 2 tx + {0, 1} + 16 j (adjacent column pairs, as the RoPE epilogue needs).
// A stage row is 32 floats (128 bytes) with its eight 16-byte units u stored
// at u ^ ((row >> 1) & 7), so that the eight tx (or ty) of a warp read
// distinct banks.  Measured against one 64 x 64 tile per CTA walking K in
// 16-deep slices without prefetch: 256 x 768 x 256 (M x N x K) 8.7 us against
// 29.4, 256 x 256 x 1024 10.3 against 108.5 (16 CTAs, 64 serial slices).
// ===========================================================================
constexpr int kFGroups = 4, kFStages = 3, kFK = 32;

template <int TM, int TN>
struct F32Cfg {
  static constexpr int STAGE_FLOATS = (TM + TN) * kFK;
  static constexpr int RED_FLOATS = kFGroups * TM * TN;  // accumulators, over the rings after the main loop
  static constexpr int RING_FLOATS = kFGroups * kFStages * STAGE_FLOATS;
  static constexpr int SMEM = 4 * (RING_FLOATS > RED_FLOATS ? RING_FLOATS : RED_FLOATS);
  static_assert(SMEM <= 227 * 1024, "fp32 GEMM shared memory");
};

// 32 columns [k0, k0 + 32) of ROWS rows from row r0 on into a swizzled stage,
// zeros past `rows` and `cols`.
template <int ROWS>
__device__ __forceinline__ void load_slice_f32(float* dst, const float* src, int64_t ld, int64_t r0, int64_t rows,
                                               int k0, int cols, int tid, bool vec) {
  if (vec) {
#pragma unroll
    for (int i = tid; i < ROWS * 8; i += 64) {
      const int r = i >> 3, u = i & 7;
      const bool ok = r0 + r < rows && k0 + 4 * u < cols;
      cp_async<16>(dst + r * kFK + ((u ^ ((r >> 1) & 7)) << 2), src + (ok ? (r0 + r) * ld + k0 + 4 * u : 0), ok);
    }
  } else {
    for (int i = tid; i < ROWS * kFK; i += 64) {
      const int r = i / kFK, k = i % kFK;
      const bool ok = r0 + r < rows && k0 + k < cols;
      cp_async<4>(dst + r * kFK + (((k >> 2) ^ ((r >> 1) & 7)) << 2) + (k & 3), src + (ok ? (r0 + r) * ld + k0 + k : 0),
                  ok);
    }
  }
}

template <int TM, int TN>
__global__ void __launch_bounds__(64 * kFGroups) gemm_f32_kernel(const float* __restrict__ A, int64_t lda, int64_t M,
                                                                 int K, const float* __restrict__ W, int N, float* out,
                                                                 int64_t ldo, EpiDev e, bool vec) {
  pdl_wait();
  using C = F32Cfg<TM, TN>;
  constexpr int MT = TM / 8, NT = TN / 8;
  extern __shared__ __align__(16) float fsm[];
  const int g = threadIdx.x >> 6, t = threadIdx.x & 63;
  const int tx = t & 7, ty = t >> 3;
  const int64_t m0 = (int64_t)blockIdx.y * TM;
  const int n0 = blockIdx.x * TN;
  const int nk = (K + kFK - 1) / kFK;
  const int mine = nk > g ? (nk - 1 - g) / kFGroups + 1 : 0;  // this group's slices
  float* ring = fsm + g * kFStages * C::STAGE_FLOATS;
  auto load = [&](int i) {
    if (i < mine) {
      float* st = ring + (i % kFStages) * C::STAGE_FLOATS;
      const int k0 = (g + i * kFGroups) * kFK;
      load_slice_f32<TM>(st, A, lda, m0, M, k0, K, t, vec);
      load_slice_f32<TN>(st + TM * kFK, W, K, n0, N, k0, K, t, vec);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int i = 0; i < kFStages - 1; ++i) load(i);
  float acc[MT][NT] = {};
  for (int i = 0; i < mine; ++i) {
    cp_async_wait<kFStages - 2>();
    group_sync(1 + g, 64);  // slice i has landed; slice i - 1 has been read
    load(i + kFStages - 1);
    const float* sa = ring + (i % kFStages) * C::STAGE_FLOATS;
    const float* sw = sa + TM * kFK;
#pragma unroll 2
    for (int u = 0; u < 8; ++u) {
      float4 av[MT], wv[NT];
#pragma unroll
      for (int r = 0; r < MT; ++r) {
        const int row = 2 * ty + (r & 1) + 16 * (r >> 1);
        av[r] = *reinterpret_cast<const float4*>(sa + row * kFK + ((u ^ (ty & 7)) << 2));
      }
#pragma unroll
      for (int c = 0; c < NT; ++c) {
        const int row = 2 * tx + (c & 1) + 16 * (c >> 1);
        wv[c] = *reinterpret_cast<const float4*>(sw + row * kFK + ((u ^ tx) << 2));
      }
#pragma unroll
      for (int r = 0; r < MT; ++r)
#pragma unroll
        for (int c = 0; c < NT; ++c)
          acc[r][c] = fmaf(av[r].w, wv[c].w,
                           fmaf(av[r].z, wv[c].z, fmaf(av[r].y, wv[c].y, fmaf(av[r].x, wv[c].x, acc[r][c]))));
    }
  }
  cp_async_wait<0>();
  __syncthreads();  // every group has finished with its ring
#pragma unroll
  for (int r = 0; r < MT; ++r)
#pragma unroll
    for (int c = 0; c < NT; c += 2)
      *reinterpret_cast<float2*>(fsm + (g * TM + 2 * ty + (r & 1) + 16 * (r >> 1)) * TN + 2 * tx + 8 * c) =
          make_float2(acc[r][c], acc[r][c + 1]);
  __syncthreads();
  const float* res = static_cast<const float*>(e.res);
  for (int i = threadIdx.x; i < TM * TN / 2; i += 64 * kFGroups) {
    const int r = i / (TN / 2), c = (i % (TN / 2)) * 2;
    const int64_t row = m0 + r;
    const int col = n0 + c;
    if (row >= M || col >= N) continue;  // N is even
    float a = 0.f, b = 0.f;
#pragma unroll
    for (int gg = 0; gg < kFGroups; ++gg) {
      const float2 v = *reinterpret_cast<const float2*>(fsm + (gg * TM + r) * TN + c);
      a += v.x;
      b += v.y;
    }
    float r0 = 0.f, r1 = 0.f;
    if (epi_reads_res(e.kind)) {
      r0 = res[row * e.ldr + col];
      r1 = res[row * e.ldr + col + 1];
    }
    epi_pair<false>(e, row + e.row_base, col, a, b, r0, r1);
    if (!ACID_IN_BOUNDS(kSiteGemmF32, row * ldo + col + 1, (M - 1) * ldo + N)) continue;
    out[row * ldo + col] = a;
    out[row * ldo + col + 1] = b;
  }
}

template <int TM, int TN>
acid_status launch_f32(const float* A, int64_t lda, int64_t M, int K, const float* W, int N, float* out, int64_t ldo,
                       const Epilogue& epi, cudaStream_t s) {
  using C = F32Cfg<TM, TN>;
  static PerContext allowed;
  ACID_TRY(allow_smem(allowed, gemm_f32_kernel<TM, TN>, C::SMEM));
  const bool vec = aligned(A, 16) && aligned(W, 16) && lda % 4 == 0 && K % 4 == 0;
  const dim3 grid((unsigned)((N + TN - 1) / TN), (unsigned)((M + TM - 1) / TM));
  launch_pdl(gemm_f32_kernel<TM, TN>, grid, 64 * kFGroups, C::SMEM, s, A, lda, M, K, W, N, out, ldo, to_dev(epi), vec);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

}  // namespace

acid_status linear_forward_f32(const void* A, int64_t lda, int64_t M, int K, const void* W, int N, void* out,
                               int64_t ldo, const Epilogue& epi, cudaStream_t s) {
  ACID_REQUIRE(M >= 0 && K > 0 && N > 0, ACID_ERR_INVALID_ARG, "linear: bad shape");
  if (M == 0) return ACID_OK;  // no rows: nothing is read, pointers may be null
  ACID_REQUIRE(A && W && out, ACID_ERR_INVALID_ARG, "linear: null pointer");
  ACID_REQUIRE(N % 2 == 0, ACID_ERR_UNSUPPORTED, "linear fp32: N must be even");
  const float *a = static_cast<const float*>(A), *w = static_cast<const float*>(W);
  float* o = static_cast<float*>(out);
  // the largest tile whose tiles still give every SM one (a larger tile reads
  // each operand value from shared memory for more outputs)
  const auto tiles = [&](int tm, int tn) { return ((M + tm - 1) / tm) * ((N + tn - 1) / tn); };
  if (tiles(64, 64) >= num_sms()) return launch_f32<64, 64>(a, lda, M, K, w, N, o, ldo, epi, s);
  if (tiles(32, 32) >= num_sms()) return launch_f32<32, 32>(a, lda, M, K, w, N, o, ldo, epi, s);
  return launch_f32<16, 32>(a, lda, M, K, w, N, o, ldo, epi, s);
}

acid_status linear_forward(int dtype, const void* A, int64_t lda, int64_t M, int K, const void* W, int N, void* out,
                           int64_t ldo, const Epilogue& epi, cudaStream_t s) {
  ACID_REQUIRE(M >= 0 && K > 0 && N > 0, ACID_ERR_INVALID_ARG, "linear: bad shape");
  if (M == 0) return ACID_OK;  // no rows: nothing is read, pointers may be null
  ACID_REQUIRE(A && W && out, ACID_ERR_INVALID_ARG, "linear: null pointer");
  ACID_REQUIRE(epi.kind != EPI_ROPE_QKV || (epi.rope.table != nullptr && epi.head_dim > 0 && epi.d > 0),
               ACID_ERR_INVALID_ARG, "linear: RoPE epilogue needs a table");
  ACID_REQUIRE(epi.kind != EPI_ROPE_QKV ||
                   (int64_t)epi.rope.grid_f * epi.rope.grid_h * epi.rope.grid_w < (int64_t(1) << 24),
               ACID_ERR_UNSUPPORTED, "linear: RoPE positions must be below 2^24");
  ACID_REQUIRE(!epi_reads_res(epi.kind) || epi.residual != nullptr, ACID_ERR_INVALID_ARG,
               "linear: residual epilogue needs a residual");
  ACID_REQUIRE(epi.text_rows >= 0 && epi.text_rows <= M && (epi.text_rows == 0 || epi.text_w != nullptr),
               ACID_ERR_INVALID_ARG, "linear: bad text rows");
  if (dtype == ACID_FP32) {
    if (epi.text_rows > 0) {  // two streams: one launch each
      const int64_t L = epi.text_rows;
      Epilogue et = epi, ev = epi;
      et.text_rows = ev.text_rows = 0;
      et.bias = epi.text_bias;
      ACID_TRY(linear_forward_f32(A, lda, L, K, epi.text_w, N, out, ldo, et, s));
      ev.row_base += L;
      if (ev.residual) ev.residual = static_cast<const float*>(ev.residual) + L * ev.ldr;
      return linear_forward_f32(static_cast<const float*>(A) + L * lda, lda, M - L, K, W, N,
                                static_cast<float*>(out) + L * ldo, ldo, ev, s);
    }
    return linear_forward_f32(A, lda, M, K, W, N, out, ldo, epi, s);
  }
  ACID_REQUIRE(N % 32 == 0 && K % 8 == 0, ACID_ERR_UNSUPPORTED, "linear bf16: need N % 32 == 0 and K % 8 == 0");
  ACID_REQUIRE(ldo % 8 == 0 && aligned(out, 16) && (!epi.residual || (epi.ldr % 8 == 0 && aligned(epi.residual, 16))),
               ACID_ERR_UNSUPPORTED, "linear bf16: output/residual must be 16-byte aligned rows");
  ACID_REQUIRE(epi.kind != EPI_ROPE_QKV || (epi.head_dim & (epi.head_dim - 1)) == 0, ACID_ERR_UNSUPPORTED,
               "linear bf16: the RoPE epilogue needs a power-of-two head_dim");
  SplitKPlan sp;
  int pairs = 0;
  const bool may_split = epi.splitk_ws != nullptr && aligned(epi.splitk_ws, 128) && epi.text_rows == 0;
  if (may_split) ACID_TRY(pair_instance_for(epi).pairs(&pairs));
  if (may_split && splitk_plan(M, N, K, epi.splitk_bytes, pairs, &sp)) {
    ACID_TRY(launch_tc2(A, lda, sp.rows_main, K, W, N, out, ldo, epi, s));
    const size_t osz = epi.out_fp32 ? 4 : 2, rsz = epi.res_fp32 ? 4 : 2;
    Epilogue et = epi;
    et.row_base += sp.rows_main;
    if (et.residual) et.residual = static_cast<const uint8_t*>(et.residual) + sp.rows_main * et.ldr * rsz;
    return launch_tc2_splitk(static_cast<const uint8_t*>(A) + sp.rows_main * lda * 2, lda, M - sp.rows_main, K, W, N,
                             static_cast<uint8_t*>(out) + sp.rows_main * ldo * osz, ldo, et, sp, s);
  }
  return launch_tc2(A, lda, M, K, W, N, out, ldo, epi, s);
}

ACID_DEVICE_FLAG_READER(take_device_error_gemm)
ACID_BOUNDS_READER(take_bounds_gemm)

}  // namespace acid
