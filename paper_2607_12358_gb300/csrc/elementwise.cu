// HBM-bound kernels of the step: drift reduction (+ fused cache apply),
// adaLN LayerNorm, GEMVs for the timestep and modulation vectors, RoPE
// tables, patchify / unpatchify + Euler update.
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace acid {

namespace {

constexpr int kThreads = 256;
constexpr int kDriftMaxBlocks = 152 * 4;  // one wave of 4 CTAs per SM on GB300

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename T> struct Vec;  // 16-byte vector of T
template <> struct Vec<__nv_bfloat16> {
  static constexpr int N = 8;
  static __device__ __forceinline__ void ld(const __nv_bfloat16* p, float* v) { load8(p, v); }
  static __device__ __forceinline__ void st(__nv_bfloat16* p, const float* v) { store8(p, v); }
};
template <> struct Vec<float> {
  static constexpr int N = 4;
  static __device__ __forceinline__ void ld(const float* p, float* v) {
    float4 a = *reinterpret_cast<const float4*>(p);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  }
  static __device__ __forceinline__ void st(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};

// One pass over prev/cur: per-thread fp32 sums of |cur - prev| and |prev|,
// fp64 across the CTA, one partial per CTA.  kApply also writes
// out = cur + resid in the same pass.  Loads are raw 16-byte vectors, U of
// them in flight per tensor and thread, unpacked after all have been issued.
template <typename T>
__device__ __forceinline__ void unpack16(const uint4& u, float* v);
template <>
__device__ __forceinline__ void unpack16<__nv_bfloat16>(const uint4& u, float* v) {
  v[0] = bf16_lo(u.x); v[1] = bf16_hi(u.x); v[2] = bf16_lo(u.y); v[3] = bf16_hi(u.y);
  v[4] = bf16_lo(u.z); v[5] = bf16_hi(u.z); v[6] = bf16_lo(u.w); v[7] = bf16_hi(u.w);
}
template <>
__device__ __forceinline__ void unpack16<float>(const uint4& u, float* v) {
  v[0] = __uint_as_float(u.x); v[1] = __uint_as_float(u.y); v[2] = __uint_as_float(u.z); v[3] = __uint_as_float(u.w);
}

template <typename T, bool kApply>
__global__ void __launch_bounds__(kThreads, 4) drift_partials_kernel(const T* __restrict__ prev,
                                                                     const T* __restrict__ cur,
                                                                     const T* __restrict__ resid, T* out,
                                                                     int64_t n, double2* __restrict__ partials) {
  pdl_wait();
  constexpr int V = Vec<T>::N;
  constexpr int U = kApply ? 2 : 4;  // 16-byte vectors in flight per thread and tensor
  const int64_t nvec = n / V;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const uint4* p4 = reinterpret_cast<const uint4*>(prev);
  const uint4* c4 = reinterpret_cast<const uint4*>(cur);
  const uint4* r4 = reinterpret_cast<const uint4*>(resid);
  float num0 = 0.f, num1 = 0.f, den0 = 0.f, den1 = 0.f;
  for (int64_t base = tid; base < nvec; base += U * stride) {
    uint4 pr[U], cr[U], rr[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = base + u * stride;
      if (i < nvec && ACID_IN_BOUNDS(kSiteDrift, i * V + V - 1, n)) {
        pr[u] = __ldcs(p4 + i);
        cr[u] = __ldcs(c4 + i);
        if (kApply) rr[u] = __ldcs(r4 + i);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = base + u * stride;
      if (i < nvec) {
        float p[V], c[V];
        unpack16<T>(pr[u], p);
        unpack16<T>(cr[u], c);
#pragma unroll
        for (int j = 0; j < V; j += 2) {
          num0 += fabsf(c[j] - p[j]);
          num1 += fabsf(c[j + 1] - p[j + 1]);
          den0 += fabsf(p[j]);
          den1 += fabsf(p[j + 1]);
        }
        if (kApply) {
          float r[V];
          unpack16<T>(rr[u], r);
#pragma unroll
          for (int j = 0; j < V; ++j) r[j] += c[j];
          Vec<T>::st(out + i * V, r);
        }
      }
    }
  }
  float num = num0 + num1, den = den0 + den1;
  for (int64_t i = nvec * V + tid; i < n; i += stride) {  // ragged tail
    const float pv = io<T>::ld(prev + i), cv = io<T>::ld(cur + i);
    num += fabsf(cv - pv);
    den += fabsf(pv);
    if (kApply) io<T>::st(out + i, cv + io<T>::ld(resid + i));
  }
  __shared__ double sn[kThreads / 32], sd[kThreads / 32];
  double dn = warp_sum_d((double)num), dd = warp_sum_d((double)den);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { sn[warp] = dn; sd[warp] = dd; }
  __syncthreads();
  if (warp == 0) {
    dn = lane < kThreads / 32 ? sn[lane] : 0.0;
    dd = lane < kThreads / 32 ? sd[lane] : 0.0;
    dn = warp_sum_d(dn);
    dd = warp_sum_d(dd);
    if (lane == 0) partials[blockIdx.x] = make_double2(dn, dd);
  }
}

// {rel, num, den} of the drift from its two sums (zero denominator: 0 when
// the numerator is 0, else +inf).
__device__ __forceinline__ void write_drift_result(double num, double den, double* result) {
  double rel;
  if (den == 0.0) rel = (num == 0.0) ? 0.0 : INFINITY;
  else rel = num / den;
  result[0] = rel;
  result[1] = num;
  result[2] = den;
}

// Fixed-order reduction of the CTA partials; result = {rel, num, den}, and the
// caller's own rel and {num, den} where given.
__global__ void __launch_bounds__(kThreads) drift_final_kernel(const double2* __restrict__ partials, int nparts,
                                                               double* result, double* rel_out, double* sums_out) {
  pdl_wait();
  double n = 0.0, d = 0.0;
  for (int i = threadIdx.x; i < nparts; i += kThreads) {
    n += partials[i].x;
    d += partials[i].y;
  }
  __shared__ double sn[kThreads / 32], sd[kThreads / 32];
  n = warp_sum_d(n);
  d = warp_sum_d(d);
  if ((threadIdx.x & 31) == 0) {
    sn[threadIdx.x >> 5] = n;
    sd[threadIdx.x >> 5] = d;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kThreads / 32; ++w) {
      sn[0] += sn[w];
      sd[0] += sd[w];
    }
    write_drift_result(sn[0], sd[0], result);
    if (rel_out != nullptr) *rel_out = result[0];
    if (sums_out != nullptr) {
      sums_out[0] = sn[0];
      sums_out[1] = sd[0];
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) add_vec_kernel(const T* __restrict__ a, const T* __restrict__ b, T* out,
                                                           int64_t n) {
  pdl_wait();
  constexpr int V = Vec<T>::N;
  const int64_t nvec = n / V;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = tid; i < nvec; i += stride) {
    if (!ACID_IN_BOUNDS(kSiteAdd, i * V + V - 1, n)) continue;
    float x[V], r[V];
    Vec<T>::ld(a + i * V, x);
    Vec<T>::ld(b + i * V, r);
#pragma unroll
    for (int j = 0; j < V; ++j) x[j] += r[j];
    Vec<T>::st(out + i * V, x);
  }
  for (int64_t i = nvec * V + tid; i < n; i += stride) io<T>::st(out + i, io<T>::ld(a + i) + io<T>::ld(b + i));
}

template <typename TA, typename TB, typename TO>
__global__ void add_mixed_kernel(const TA* __restrict__ a, const TB* __restrict__ b, TO* out, int64_t n, float bs) {
  pdl_wait();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    io<TO>::st(out + i, io<TA>::ld(a + i) + bs * io<TB>::ld(b + i));
}

// The same on eight consecutive values per thread (16-byte aligned operands);
// READ_B false: out = a (b_scale 0, b not read).
template <typename TA, typename TB, typename TO, bool READ_B>
__global__ void add_mixed8_kernel(const TA* __restrict__ a, const TB* __restrict__ b, TO* out, int64_t n, float bs) {
  pdl_wait();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t i = tid; i < n / 8; i += stride) {
    if (!ACID_IN_BOUNDS(kSiteAdd, 8 * i + 7, n)) continue;
    float x[8];
    load8(a + 8 * i, x);
    if constexpr (READ_B) {
      float y[8];
      load8(b + 8 * i, y);
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = x[j] + bs * y[j];
    }
    store8(out + 8 * i, x);
  }
  for (int64_t i = n / 8 * 8 + tid; i < n; i += stride)
    io<TO>::st(out + i, READ_B ? io<TA>::ld(a + i) + bs * io<TB>::ld(b + i) : io<TA>::ld(a + i));
}

// 1D bulk copies from global to shared memory (16-byte aligned, sizes multiples
// of 16).
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// The same with an L2 cache policy for the source lines.
__device__ __forceinline__ void bulk_load_hint(void* dst, const void* src, uint32_t bytes, uint64_t* bar,
                                               uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// ---------------------------------------------------------------- LayerNorm
// Both kernels keep a row in registers and run the two-pass statistics and the
// modulation on packed fp32 pairs, unpacked once and centred in place.
// four values of a row
__device__ __forceinline__ void load_quad(const __nv_bfloat16* p, uint64_t* v) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  v[0] = f2_pack(bf16_lo(u.x), bf16_hi(u.x));
  v[1] = f2_pack(bf16_lo(u.y), bf16_hi(u.y));
}
__device__ __forceinline__ void load_quad(const float* p, uint64_t* v) {
  const float4 u = *reinterpret_cast<const float4*>(p);
  v[0] = f2_pack(u.x, u.y);
  v[1] = f2_pack(u.z, u.w);
}
// a pair rounded to T
template <typename T>
__device__ __forceinline__ uint64_t round_to(uint64_t v) {
  if constexpr (sizeof(T) == 2) {
    float a, b;
    f2_unpack(v, a, b);
    const uint32_t w = pack_bf16(a, b);
    return f2_pack(bf16_lo(w), bf16_hi(w));
  } else {
    return v;
  }
}
__device__ __forceinline__ void store_quad(__nv_bfloat16* p, const uint64_t* v) {
  float a, b, c, d;
  f2_unpack(v[0], a, b);
  f2_unpack(v[1], c, d);
  *reinterpret_cast<uint2*>(p) = make_uint2(pack_bf16(a, b), pack_bf16(c, d));
}
__device__ __forceinline__ void store_quad(float* p, const uint64_t* v) {
  float a, b, c, d;
  f2_unpack(v[0], a, b);
  f2_unpack(v[1], c, d);
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}

// v holds a lane's quads (columns (i * 32 + lane) * 4 ..) of a warp's row, zeros
// past d: centres them in place and returns 1 / sqrt(var + eps).
template <int NV, bool FULL>
__device__ __forceinline__ float row_center(uint64_t (&v)[NV][2], int lane, int d, float eps) {
  uint64_t s[2] = {}, t[2] = {};
#pragma unroll
  for (int i = 0; i < NV; ++i)
#pragma unroll
    for (int q = 0; q < 2; ++q) s[q] = f2_add(s[q], v[i][q]);
  float a, b;
  f2_unpack(f2_add(s[0], s[1]), a, b);
  const float mean = warp_sum_f(a + b) / d;
  const uint64_t nm = f2_pack(-mean, -mean);
#pragma unroll
  for (int i = 0; i < NV; ++i)
    if (FULL || (i * 32 + lane) * 4 < d) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        v[i][q] = f2_add(v[i][q], nm);
        t[q] = f2_fma(v[i][q], v[i][q], t[q]);
      }
    }
  f2_unpack(f2_add(t[0], t[1]), a, b);
  return rsqrtf(warp_sum_f(a + b) / d + eps);
}

// What a row kernel does beside the LayerNorm of x.
enum LnMode : int {
  kLnPlain = 0,
  kLnReuse = 1,  // x = h + r first, rounded to TX (the reused step's state)
  kLnResid = 2   // also r = x - h (the computed step's residual)
};

struct LnArgs {
  const void* x;
  void* y;
  const float* h;       // kLnReuse, kLnResid: the stack's input
  float* r;             // kLnReuse: read, kLnResid: written
  int64_t rows, split;  // rows below split take the text vectors
  int d, vecs;          // vecs: modulation streams (0, 1 video only, 2 video and text)
  const float *shv, *scv, *sht, *sct;
  float eps;
};

// Rows of up to 512 columns: one warp per row, straight from and to global memory.  A lane
// holds four consecutive columns in every 128, so that its loads and stores
// of bf16 (8 bytes) and fp32 (16 bytes) rows and vectors are contiguous over the
// warp.
constexpr int kLnThreads = 128;

// FULL: the row fills every lane (d = 128 NV).  The cached residual of a
// TeaCache step is applied (kLnReuse) or stored (kLnResid) in the same pass:
// apart, the state was written and read again, or read a second time.
template <typename Tin, typename Tout, int NV, bool FULL, int MODE>
__global__ void __launch_bounds__(kLnThreads, 5) ln_mod_rows_kernel(LnArgs a) {
  pdl_wait();
  const int64_t row = ((int64_t)blockIdx.x * kLnThreads + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, d = a.d;
  if (row >= a.rows) return;
  const Tin* xr = static_cast<const Tin*>(a.x) + row * d;
  Tout* yr = static_cast<Tout*>(a.y) + row * d;
  uint64_t v[NV][2];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int c = (i * 32 + lane) * 4;
    if (!FULL || kBoundsChecked) v[i][0] = v[i][1] = 0;
    if (!((FULL || c < d) && ACID_IN_BOUNDS(kSiteLayerNorm, row * d + c + 3, a.rows * d))) continue;
    if constexpr (MODE == kLnReuse) {
      uint64_t r[2];
      load_quad(a.h + row * d + c, v[i]);
      load_quad(a.r + row * d + c, r);
      v[i][0] = round_to<Tin>(f2_add(v[i][0], r[0]));
      v[i][1] = round_to<Tin>(f2_add(v[i][1], r[1]));
    } else {
      load_quad(xr + c, v[i]);
    }
    if constexpr (MODE == kLnResid) {
      const float4 h = *reinterpret_cast<const float4*>(a.h + row * d + c);
      float x0, x1, x2, x3;
      f2_unpack(v[i][0], x0, x1);
      f2_unpack(v[i][1], x2, x3);
      *reinterpret_cast<float4*>(a.r + row * d + c) = make_float4(x0 - h.x, x1 - h.y, x2 - h.z, x3 - h.w);
    }
  }
  const float rstd = row_center<NV, FULL>(v, lane, d, a.eps);
  const uint64_t rs = f2_pack(rstd, rstd);
  const bool text = a.vecs == 2 && row < a.split;
  const float *sc = text ? a.sct : a.scv, *sh = text ? a.sht : a.shv;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int c = (i * 32 + lane) * 4;
    if (!FULL && c >= d) continue;
    v[i][0] = f2_mul(v[i][0], rs);
    v[i][1] = f2_mul(v[i][1], rs);
    if (a.vecs) {
      const float4 p = *reinterpret_cast<const float4*>(sc + c), q = *reinterpret_cast<const float4*>(sh + c);
      v[i][0] = f2_fma(v[i][0], f2_pack(1.f + p.x, 1.f + p.y), f2_pack(q.x, q.y));
      v[i][1] = f2_fma(v[i][1], f2_pack(1.f + p.z, 1.f + p.w), f2_pack(q.z, q.w));
    }
    if (ACID_IN_BOUNDS(kSiteLayerNorm, row * d + c + 3, a.rows * d)) store_quad(yr + c, v[i]);
  }
}

// Rows of more than 512 columns: persistent CTAs of four warps, a row at a
// time.  One thread streams the CTA's next rows into a shared-memory ring with
// bulk copies; a lane keeps NQ quads of the row and of its modulation (1 + scale,
// shift) in registers, so that the vectors are read once per CTA and stream and
// not once per row, and a row's serial chain (read, two reductions, store) is
// a fraction of what one warp makes of it.  HBM bounds large row counts, the
// rows' chains small ones.  Measured (us, one warp a row -> this): 4846 x 3072
// bf16 11.0 -> 9.1, 9000 x 3072 bf16 26.6 -> 17.0, 17776 x 1920 bf16 25.4 -> 21.2,
// 50000 x 3072 fp32 to bf16 158 -> 142.  A reused step's pass over 7800 x 1536:
// 20.5 -> 15.4.
constexpr int kLnMaxStages = 4;
// CTAs per SM: 16 to 18 warps, as many as the registers of a lane's quads and
// their modulation leave room for.
template <int WPR>
constexpr int kLnCtas = WPR == 3 ? 6 : 16 / WPR;

template <typename Tin, typename Tout, int WPR, int NQ, bool FULL, int MODE>
__global__ void __launch_bounds__(32 * WPR, kLnCtas<WPR>) ln_mod_team_kernel(LnArgs a, int stages) {
  extern __shared__ __align__(128) uint8_t lsm[];
  constexpr int kTeam = 32 * WPR;
  __shared__ __align__(16) float red[2][4];
  __shared__ uint64_t full[kLnMaxStages];
  __shared__ int gave_up;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, d = a.d;
  using T0 = std::conditional_t<MODE == kLnReuse, float, Tin>;
  const T0* src0 = static_cast<const T0*>(MODE == kLnReuse ? (const void*)a.h : a.x);
  const float* src1 = MODE == kLnReuse ? a.r : a.h;
  const uint32_t bytes0 = d * (uint32_t)sizeof(T0), bytes1 = MODE == kLnPlain ? 0 : d * 4u;
  const int64_t mine = blockIdx.x < a.rows ? (a.rows - 1 - blockIdx.x) / gridDim.x + 1 : 0;
  auto issue = [&](int64_t k, int st) {
    int64_t row = blockIdx.x + k * gridDim.x;
    if (!ACID_IN_BOUNDS(kSiteLayerNorm, row, a.rows)) row = 0;  // (debug builds) read row 0 instead
    uint8_t* dst = lsm + (size_t)st * (bytes0 + bytes1);
    mbar_expect_tx(&full[st], bytes0 + bytes1);
    bulk_load(dst, src0 + row * d, bytes0, &full[st]);
    if constexpr (MODE != kLnPlain) bulk_load(dst + bytes0, src1 + row * d, bytes1, &full[st]);
  };
  if (tid < 8) red[tid >> 2][tid & 3] = 0.f;
  if (tid == 0) {
    gave_up = 0;
    for (int i = 0; i < stages; ++i) mbar_init(&full[i], 1);
    mbar_fence_init();
  }
  pdl_wait();
  if (tid == 0)
    for (int k = 0; k < mine && k < stages; ++k) issue(k, k);
  uint64_t sc[NQ][2], sh[NQ][2];
  auto load_mod = [&](const float* scp, const float* shp) {
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const int c = (i * kTeam + tid) * 4;
      if (!FULL && c >= d) continue;
      const float4 p = *reinterpret_cast<const float4*>(scp + c), q = *reinterpret_cast<const float4*>(shp + c);
      sc[i][0] = f2_pack(1.f + p.x, 1.f + p.y);
      sc[i][1] = f2_pack(1.f + p.z, 1.f + p.w);
      sh[i][0] = f2_pack(q.x, q.y);
      sh[i][1] = f2_pack(q.z, q.w);
    }
  };
  bool text = a.vecs == 2 && blockIdx.x < a.split;
  if (a.vecs) load_mod(text ? a.sct : a.scv, text ? a.sht : a.shv);
  __syncthreads();
  // the sum over the CTA of each warp's share
  auto team_sum = [&](uint64_t s, float* r) {
    float x, y;
    f2_unpack(s, x, y);
    x = warp_sum_f(x + y);
    if (lane == 0) r[warp] = x;
    __syncthreads();
    const float4 t = *reinterpret_cast<const float4*>(r);
    return (t.x + t.y) + (t.z + t.w);
  };
  int st = 0;
  uint32_t phase = 0;
  auto next = [&] {
    if (++st == stages) {
      st = 0;
      phase ^= 1;
    }
  };
  int64_t k = 0, row = blockIdx.x;
  for (; k < mine; ++k, row += gridDim.x, next()) {
    if (!mbar_wait(&full[st], phase)) gave_up = 1;
    const uint8_t* buf = lsm + (size_t)st * (bytes0 + bytes1);
    const T0* r0 = reinterpret_cast<const T0*>(buf);
    const float* r1 = reinterpret_cast<const float*>(buf + bytes0);
    uint64_t v[NQ][2], s = 0, t = 0;
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const int c = (i * kTeam + tid) * 4;
      v[i][0] = v[i][1] = 0;
      if (!FULL && c >= d) continue;
      load_quad(r0 + c, v[i]);
      if constexpr (MODE == kLnReuse) {
        uint64_t r[2];
        load_quad(r1 + c, r);
        v[i][0] = round_to<Tin>(f2_add(v[i][0], r[0]));
        v[i][1] = round_to<Tin>(f2_add(v[i][1], r[1]));
      }
      if constexpr (MODE == kLnResid) {
        const float4 h = *reinterpret_cast<const float4*>(r1 + c);
        float x0, x1, x2, x3;
        f2_unpack(v[i][0], x0, x1);
        f2_unpack(v[i][1], x2, x3);
        if (ACID_IN_BOUNDS(kSiteLayerNorm, row * d + c + 3, a.rows * d))
          *reinterpret_cast<float4*>(a.r + row * d + c) = make_float4(x0 - h.x, x1 - h.y, x2 - h.z, x3 - h.w);
      }
      s = f2_add(s, f2_add(v[i][0], v[i][1]));
    }
    const float mean = team_sum(s, red[0]) / d;
    if (gave_up) break;  // a wait ran out: the CTA leaves together
    if (tid == 0 && k + stages < mine) issue(k + stages, st);  // every lane holds its values
    const uint64_t nm = f2_pack(-mean, -mean);
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      if (!FULL && (i * kTeam + tid) * 4 >= d) continue;
      v[i][0] = f2_add(v[i][0], nm);
      v[i][1] = f2_add(v[i][1], nm);
      t = f2_fma(v[i][0], v[i][0], t);
      t = f2_fma(v[i][1], v[i][1], t);
    }
    // a warp writes red[0] of the next row behind this barrier, red[1] behind the next row's first
    const float rstd = rsqrtf(team_sum(t, red[1]) / d + a.eps);
    const uint64_t rs = f2_pack(rstd, rstd);
    if (text && row >= a.split) {
      text = false;
      load_mod(a.scv, a.shv);
    }
    Tout* yr = static_cast<Tout*>(a.y) + row * d;
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const int c = (i * kTeam + tid) * 4;
      if (!FULL && c >= d) continue;
      v[i][0] = f2_mul(v[i][0], rs);
      v[i][1] = f2_mul(v[i][1], rs);
      if (a.vecs) {
        v[i][0] = f2_fma(v[i][0], sc[i][0], sh[i][0]);
        v[i][1] = f2_fma(v[i][1], sc[i][1], sh[i][1]);
      }
      if (ACID_IN_BOUNDS(kSiteLayerNorm, row * d + c + 3, a.rows * d)) store_quad(yr + c, v[i]);
    }
  }
  // after a wait ran out: the copies already issued land before the CTA exits
  if (tid == 0)
    for (int64_t j = k; j < mine && j < k + stages; ++j, next()) mbar_wait(&full[st], phase);
}

// ------------------------------------------- TEMNI drift from two H_in rows
// The sums |TEMNI_t - TEMNI_{t-1}| and |TEMNI_{t-1}| of the TeaCache signal,
// with TEMNI = LN(H_in) (1 + scale) + shift at each step's own (shift,
// scale).  Both TEMNI rows are formed in registers from the fp32 patch
// embeddings H_in_t (xc) and H_in_{t-1} (xp), so the kernel reads 8 bytes per
// element and writes nothing but one fp64 partial pair per CTA (reduced by
// drift_final_kernel, or with a done counter by the CTA that finishes last).
// A group of WPR warps takes one row pair at a time (rows counted from the
// end: g, g + total groups, ... from the last row down) and streams its row pairs
// into its own two-stage shared-memory ring with 1D bulk copies (completion
// counted on the stage's mbarrier), so the bytes in flight come from shared
// memory, not registers; a lane keeps its NV4 x 4 columns of both rows in
// registers after one read of the stage, which is refilled as soon as the
// group has read it.  Long rows leave shared memory for few groups (three at
// 3072 columns), so several warps share a row: with one warp each, three warps
// per SM did all the arithmetic (16000 x 3072: 122 us).  The four modulation
// vectors (shift and 1 + scale of both steps) are staged once per CTA in
// shared memory.  Row statistics: mean and variance from sums of (x - K) and
// (x - K)^2 with K the row's first element, which keeps the fp32 cancellation
// small (K lies within a few standard deviations of the mean), by warp shuffles
// and, across a group's warps, through shared memory.  Step 0 gives zero sums.
constexpr int kTemniStages = 2;
constexpr int kTemniMaxWarps = 16, kTemniMaxGroups = 8;

template <int NV4, int WPR>
__global__ void __launch_bounds__(32 * (WPR == 1 ? kTemniMaxGroups : kTemniMaxWarps), 1)
    temni_drift_kernel(const float* __restrict__ xc, const float* __restrict__ xp, const int* step_dev, int step_host,
                       int64_t rows, int d, const float* __restrict__ shc, const float* __restrict__ scc,
                       const float* __restrict__ shp, const float* __restrict__ scp, float eps,
                       double2* __restrict__ partials, unsigned int* done, double* result) {
  pdl_wait();
  extern __shared__ __align__(128) uint8_t tsm[];
  const int nwarps = blockDim.x >> 5, ngroups = nwarps / WPR;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = warp / WPR, wg = warp % WPR;  // group, warp in the group
  // four d-long vectors: shift_c, 1 + scale_c, shift_p, 1 + scale_p (separate
  // arrays, so that a warp's 16-byte reads of one vector are contiguous)
  float4* mod = reinterpret_cast<float4*>(tsm);
  float* ring = reinterpret_cast<float*>(tsm + (size_t)16 * d);                                   // [group][stage][2][d]
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + (size_t)ngroups * kTemniStages * 2 * d);    // [group][stage]
  __shared__ double rd[2][kTemniMaxWarps];
  __shared__ float4 stats[2][kTemniMaxWarps];  // partial row sums, by row parity
  const int step = step_dev ? *step_dev : step_host;
  float* wr = ring + (size_t)grp * kTemniStages * 2 * d;
  uint64_t* wf = full + grp * kTemniStages;
  const int64_t gw = (int64_t)blockIdx.x * ngroups + grp, nw = (int64_t)gridDim.x * ngroups;
  const int64_t n_my = (step > 0 && gw < rows) ? (rows - 1 - gw) / nw + 1 : 0;
  const uint32_t row_bytes = (uint32_t)d * sizeof(float);
  const bool leader = wg == 0 && lane == 0;
  // Rows from the last one down: the patch embedding that writes h_cur just
  // before this kernel leaves its last rows in L2 (dirty), so they are read
  // first.  The previous step's rows are not read again in this step: they
  // are loaded evict-first, so that they, and not those dirty h_cur lines,
  // give way to new lines, and no write-back of h_cur falls into this kernel.
  const uint64_t prev_policy = l2_policy_evict_first();
  auto issue = [&](int64_t k) {
    const int st = (int)(k % kTemniStages);
    int64_t row = rows - 1 - (gw + k * nw);
    if (!ACID_IN_BOUNDS(kSiteTemni, row, rows)) row = 0;  // (debug builds) read row 0 instead
    mbar_expect_tx(&wf[st], 2 * row_bytes);
    bulk_load(wr + (size_t)st * 2 * d, xc + row * d, row_bytes, &wf[st]);
    bulk_load_hint(wr + (size_t)st * 2 * d + d, xp + row * d, row_bytes, &wf[st], prev_policy);
  };
  // each group's first copies are issued before the modulation vectors are
  // staged, so their latency overlaps the staging
  if (leader) {
    for (int i = 0; i < kTemniStages; ++i) mbar_init(&wf[i], 1);
    mbar_fence_init();
    for (int64_t k = 0; k < n_my && k < kTemniStages; ++k) issue(k);
  }
  for (int i = threadIdx.x; i < d / 4; i += blockDim.x) {
    const float4 a = reinterpret_cast<const float4*>(shc)[i], b = reinterpret_cast<const float4*>(scc)[i];
    const float4 c = reinterpret_cast<const float4*>(shp)[i], e = reinterpret_cast<const float4*>(scp)[i];
    const int q = d / 4;
    mod[i] = a;
    mod[q + i] = make_float4(1.f + b.x, 1.f + b.y, 1.f + b.z, 1.f + b.w);
    mod[2 * q + i] = c;
    mod[3 * q + i] = make_float4(1.f + e.x, 1.f + e.y, 1.f + e.z, 1.f + e.w);
  }
  __syncthreads();  // modulation vectors staged, barriers initialised
  const float inv_d = 1.0f / d;
  float num = 0.f, den = 0.f;
  int64_t k = 0;
  for (; k < n_my; ++k) {
    const int st = (int)(k % kTemniStages);
    const bool ok = __all_sync(0xffffffffu, mbar_wait(&wf[st], (uint32_t)((k / kTemniStages) & 1)));
    if (WPR == 1 && !ok) break;
    const float4* rc = reinterpret_cast<const float4*>(wr + (size_t)st * 2 * d);
    const float4* rp = rc + d / 4;
    // lane's vectors: (i * WPR + wg) * 32 + lane, i < NV4 (4 columns each)
    float4 cv[NV4], pv[NV4];
    const float kc = wr[(size_t)st * 2 * d], kp = wr[(size_t)st * 2 * d + d];  // shifts: the rows' first elements
    float s1c = 0.f, s2c = 0.f, s1p = 0.f, s2p = 0.f;
#pragma unroll
    for (int i = 0; i < NV4; ++i) {
      const int v = (i * WPR + wg) * 32 + lane;
      if (v < d / 4) {
        const float4 c = rc[v], p = rp[v];
        cv[i] = c;
        pv[i] = p;
        const float c0 = c.x - kc, c1 = c.y - kc, c2 = c.z - kc, c3 = c.w - kc;
        const float p0 = p.x - kp, p1 = p.y - kp, p2 = p.z - kp, p3 = p.w - kp;
        s1c += (c0 + c1) + (c2 + c3);
        s2c = fmaf(c0, c0, fmaf(c1, c1, fmaf(c2, c2, fmaf(c3, c3, s2c))));
        s1p += (p0 + p1) + (p2 + p3);
        s2p = fmaf(p0, p0, fmaf(p1, p1, fmaf(p2, p2, fmaf(p3, p3, s2p))));
      }
    }
    if constexpr (WPR == 1) {
      __syncwarp();
      if (lane == 0 && k + kTemniStages < n_my) issue(k + kTemniStages);  // every lane holds its values
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s1c += __shfl_xor_sync(0xffffffffu, s1c, o);
      s2c += __shfl_xor_sync(0xffffffffu, s2c, o);
      s1p += __shfl_xor_sync(0xffffffffu, s1p, o);
      s2p += __shfl_xor_sync(0xffffffffu, s2p, o);
    }
    if constexpr (WPR > 1) {
      // the sums of row k + 2 overwrite these behind the barrier of row k + 1
      if (lane == 0) stats[k & 1][warp] = make_float4(s1c, s2c, s1p, s2p);
      if (!group_all(1 + grp, 32 * WPR, ok)) break;  // a wait of one of its warps ran out: the group leaves together
      if (leader && k + kTemniStages < n_my) issue(k + kTemniStages);  // the whole group holds its values
      s1c = s2c = s1p = s2p = 0.f;
#pragma unroll
      for (int w = 0; w < WPR; ++w) {
        const float4 t = stats[k & 1][grp * WPR + w];
        s1c += t.x;
        s2c += t.y;
        s1p += t.z;
        s2p += t.w;
      }
    }
    const float dc = s1c * inv_d, dp = s1p * inv_d;  // mean - K
    const float mc = kc + dc, mp = kp + dp;
    const float rsc = rsqrtf(fmaxf(s2c * inv_d - dc * dc, 0.f) + eps);
    const float rsp = rsqrtf(fmaxf(s2p * inv_d - dp * dp, 0.f) + eps);
#pragma unroll
    for (int i = 0; i < NV4; ++i) {
      const int v = (i * WPR + wg) * 32 + lane;
      if (v < d / 4) {
        const float4 c = cv[i], p = pv[i];
        const int q = d / 4;
        const float4 bcv = mod[v], acv = mod[q + v], bpv = mod[2 * q + v], apv = mod[3 * q + v];
        const float cc[4] = {c.x, c.y, c.z, c.w}, pp[4] = {p.x, p.y, p.z, p.w};
        const float ac[4] = {acv.x, acv.y, acv.z, acv.w}, bc[4] = {bcv.x, bcv.y, bcv.z, bcv.w};
        const float ap[4] = {apv.x, apv.y, apv.z, apv.w}, bp[4] = {bpv.x, bpv.y, bpv.z, bpv.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float uc = fmaf((cc[j] - mc) * rsc, ac[j], bc[j]);
          const float up = fmaf((pp[j] - mp) * rsp, ap[j], bp[j]);
          num += fabsf(uc - up);
          den += fabsf(up);
        }
      }
    }
  }
  // after a wait ran out: the copies already issued land before the CTA exits
  if (k < n_my && leader)
    for (int64_t j = k; j < n_my && j < k + kTemniStages; ++j)
      mbar_wait(&wf[j % kTemniStages], (uint32_t)((j / kTemniStages) & 1));
  double dn = warp_sum_d((double)num), dd = warp_sum_d((double)den);
  if (lane == 0) {
    rd[0][warp] = dn;
    rd[1][warp] = dd;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    dn = 0.0;
    dd = 0.0;
    for (int w = 0; w < nwarps; ++w) {
      dn += rd[0][w];
      dd += rd[1][w];
    }
    partials[blockIdx.x] = make_double2(dn, dd);
  }
  // With a done counter (zero on entry), the CTA that finishes last sums the
  // partials in a fixed order and writes the result, then sets the counter
  // back to zero: no second launch.
  if (done != nullptr) {
    __shared__ bool last;
    if (threadIdx.x == 0) {
      __threadfence();  // this CTA's partial is visible before it is counted
      last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (last && warp == 0) {
      __threadfence();
      double n = 0.0, e = 0.0;
      for (int i = lane; i < (int)gridDim.x; i += 32) {
        const double2 p = __ldcg(&partials[i]);
        n += p.x;
        e += p.y;
      }
      n = warp_sum_d(n);
      e = warp_sum_d(e);
      if (lane == 0) {
        write_drift_result(n, e, result);
        *done = 0u;
      }
    }
  }
}

// ---------------------------------------------------------------- GEMV
// A warp forms R outputs of one or two matrices that share the input (rows
// from n_out on are the second's).  The input is staged once per CTA, as two
// arrays of alternating 16-byte units, so that the warp's reads of its eight
// values per lane are contiguous, and each read serves R weight rows: with one
// row per warp and a 32-byte lane stride the shared-memory reads took four
// times the cycles of the weight stream.
struct GemvMat {
  const void* W;
  const float* b;
  float* y;
  int n_out;
};

template <typename TW, int R>
__global__ void __launch_bounds__(kThreads, 3) gemv_kernel(GemvMat m0, GemvMat m1, const float* __restrict__ x, int k,
                                                           int silu_in) {
  pdl_wait();
  extern __shared__ __align__(16) float xs[];  // [2][k / 2]: columns 8 i + {0..3}, then 8 i + {4..7}
  for (int i = threadIdx.x; i < k; i += kThreads) {
    const float v = x[i];
    xs[(i & 4 ? k / 2 : 0) + (i >> 3) * 4 + (i & 3)] = silu_in ? silu(v) : v;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int total = m0.n_out + m1.n_out;
  for (int first = (blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * R; first < total;
       first += gridDim.x * (kThreads / 32) * R) {
    const TW* wr[R];
    float acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = min(first + r, total - 1);  // rows past the end repeat the last one and are not stored
      wr[r] = row < m0.n_out ? static_cast<const TW*>(m0.W) + (int64_t)row * k
                             : static_cast<const TW*>(m1.W) + (int64_t)(row - m0.n_out) * k;
      acc[r] = 0.f;
    }
#pragma unroll(8 / R)
    for (int c = lane * 8; c < k; c += 256) {
      if (!ACID_IN_BOUNDS(kSiteGemv, c + 7, k)) continue;
      float w[R][8];
#pragma unroll
      for (int r = 0; r < R; ++r) load8(wr[r] + c, w[r]);
      const float4 lo = *reinterpret_cast<const float4*>(xs + c / 2);
      const float4 hi = *reinterpret_cast<const float4*>(xs + k / 2 + c / 2);
      const float xv[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[r] = fmaf(w[r][j], xv[j], acc[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = warp_sum_f(acc[r]);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = first + r;
      if (lane == 0 && row < total) {
        const GemvMat& m = row < m0.n_out ? m0 : m1;
        const int o = row < m0.n_out ? row : row - m0.n_out;
        m.y[o] = acc[r] + (m.b ? m.b[o] : 0.f);
      }
    }
  }
}

// Small fp64 tables.  An SM has few fp64 units, so these run as many CTAs of
// one warp, spread over the SMs, with the cosines and sines in separate warps:
// 128 frequencies as one CTA of 128 threads took 5.6 us, a 1200-entry RoPE
// table on 10 CTAs 8 us.
constexpr int kTableThreads = 32;

__device__ __forceinline__ void sinusoid_at(float* out, double t, int half, int j) {
  const double a = t * exp(-log(10000.0) * (double)j / (double)half);
  if (blockIdx.y == 0)
    out[j] = (float)cos(a);
  else
    out[half + j] = (float)sin(a);
}

__global__ void sinusoid_kernel(float* out, double t, int half) {
  pdl_wait();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < half) sinusoid_at(out, t, half, j);
}

// t = 1000 sigma[step] with the step index read from device memory
__global__ void sinusoid_sig_kernel(float* out, const double* sig, const int* step, int half) {
  pdl_wait();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < half) sinusoid_at(out, 1000.0 * sig[*step], half, j);
}

__global__ void rope_table_kernel(float2* tbl, int F, int H, int W, int pt, int ph, int pw, double theta) {
  pdl_wait();
  // pt / ph / pw: rotation pairs per axis (t, h, w)
  const int64_t total = (int64_t)F * pt + (int64_t)H * ph + (int64_t)W * pw;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  int64_t r = i;
  int pos, j, pairs;
  if (r < (int64_t)F * pt) {
    pos = (int)(r / pt); j = (int)(r % pt); pairs = pt;
  } else if ((r -= (int64_t)F * pt) < (int64_t)H * ph) {
    pos = (int)(r / ph); j = (int)(r % ph); pairs = ph;
  } else {
    r -= (int64_t)H * ph;
    pos = (int)(r / pw); j = (int)(r % pw); pairs = pw;
  }
  const double dim = 2.0 * pairs;
  const double ang = (double)pos * pow(theta, -2.0 * j / dim);
  if (blockIdx.y == 0)
    tbl[i].x = (float)cos(ang);
  else
    tbl[i].y = (float)sin(ang);
}

// ---------------------------------------------------------------- patches
// One CTA moves the tokens of up to 32 patches along a latent row: rows of the
// latent in and token vectors out (or back), both contiguous, through a
// shared-memory tile [patch][P].  Element by element in token order the
// latent accesses covered 8 bytes a line, behind six 64-bit divisions each.
// Patch vectors of more than kPatchMaxP values take the element kernels below.
constexpr int kPatchTile = 32, kPatchMaxP = 256;

struct PatchGeo {
  int C, F, H, W, pt, ph, pw;
};
// The tile of this CTA (blockIdx.x: tile along the row, y: patch row, z:
// frame): its first token, its patch count, and element e of it: shared index,
// latent index.
struct PatchTile {
  PatchGeo g;
  int w0, nw, P;
  int64_t n0;
  __device__ __forceinline__ explicit PatchTile(const PatchGeo& geo) : g(geo) {
    const int Wp = g.W / g.pw;
    w0 = blockIdx.x * kPatchTile;
    nw = min(kPatchTile, Wp - w0);
    P = g.C * g.pt * g.ph * g.pw;
    n0 = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * Wp + w0;
  }
  // e counts latent row by latent row: r = (c, dt, dh), then nw * pw columns
  __device__ __forceinline__ void at(int e, int& sidx, int64_t& lidx) const {
    const int cols = nw * g.pw, r = e / cols, x = e - r * cols;
    const int dh = r % g.ph, q = r / g.ph, dt = q % g.pt, c = q / g.pt;
    const int tok = x / g.pw;
    sidx = tok * (P + 1) + r * g.pw + (x - tok * g.pw);
    lidx = (((int64_t)c * g.F + (int)blockIdx.z * g.pt + dt) * g.H + (int)blockIdx.y * g.ph + dh) * g.W + w0 * g.pw + x;
  }
};

// SPLIT: bf16 tokens of width 2P that carry each fp32 value as the sum of two
// bf16 parts: hi = bf16(x) in column p, lo = bf16(x - hi) in column P + p.
// x - hi is exact in fp32 and lo rounds it to 8 bits, so hi + lo equals x to
// within 2^-17 |x|; a bf16 GEMM against the weights repeated along K ([W | W])
// then forms the fp32-input patch embedding on tensor cores.  Otherwise fp32
// tokens.
template <bool SPLIT>
__global__ void __launch_bounds__(kThreads) patchify_tile_kernel(const float* __restrict__ lat, void* tok,
                                                                 PatchGeo geo) {
  pdl_wait();
  extern __shared__ float tile[];
  const PatchTile t(geo);
  const int n = t.nw * t.P;
  for (int e = threadIdx.x; e < n; e += kThreads) {
    int si;
    int64_t li;
    t.at(e, si, li);
    tile[si] = ACID_IN_BOUNDS(kSitePatchify, li, (int64_t)geo.C * geo.F * geo.H * geo.W) ? lat[li] : 0.f;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n; e += kThreads) {
    const int k = e / t.P, p = e - k * t.P;
    const float x = tile[k * (t.P + 1) + p];
    if constexpr (SPLIT) {
      __nv_bfloat16* o = static_cast<__nv_bfloat16*>(tok) + (t.n0 + k) * 2 * t.P + p;
      const __nv_bfloat16 hi = __float2bfloat16_rn(x);
      o[0] = hi;
      o[t.P] = __float2bfloat16_rn(x - __bfloat162float(hi));
    } else {
      static_cast<float*>(tok)[(t.n0 + k) * t.P + p] = x;
    }
  }
}

__global__ void __launch_bounds__(kThreads) unpatchify_tile_kernel(const float* __restrict__ vtok,
                                                                   float* __restrict__ vout, float* lat, PatchGeo geo,
                                                                   float dsig) {
  pdl_wait();
  extern __shared__ float tile[];
  const PatchTile t(geo);
  const int n = t.nw * t.P;
  for (int e = threadIdx.x; e < n; e += kThreads) {
    const int k = e / t.P;
    tile[k * (t.P + 1) + (e - k * t.P)] = vtok[t.n0 * t.P + e];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n; e += kThreads) {
    int si;
    int64_t li;
    t.at(e, si, li);
    if (!ACID_IN_BOUNDS(kSiteUnpatchify, li, (int64_t)geo.C * geo.F * geo.H * geo.W)) continue;
    const float v = tile[si];
    if (vout) vout[li] = v;
    if (lat) lat[li] = fmaf(dsig, v, lat[li]);
  }
}

__global__ void patchify_kernel(const float* __restrict__ lat, float* __restrict__ tok, int C, int F, int H, int W,
                                int pt, int ph, int pw) {
  pdl_wait();
  const int Hp = H / ph, Wp = W / pw;
  const int P = C * pt * ph * pw;
  const int64_t total = (int64_t)(F / pt) * Hp * Wp * P;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
    const int64_t n = i / P;
    int p = (int)(i % P);
    const int f = (int)(n / ((int64_t)Hp * Wp)), h = (int)((n / Wp) % Hp), w = (int)(n % Wp);
    const int dw = p % pw; p /= pw;
    const int dh = p % ph; p /= ph;
    const int dt = p % pt; p /= pt;
    const int c = p;
    const int64_t src = (((int64_t)c * F + (f * pt + dt)) * H + (h * ph + dh)) * W + (w * pw + dw);
    if (ACID_IN_BOUNDS(kSitePatchify, src, (int64_t)C * F * H * W)) tok[i] = lat[src];
  }
}

// The same as hi and lo bf16 parts (see patchify_tile_kernel).
__global__ void patchify_split_kernel(const float* __restrict__ lat, __nv_bfloat16* __restrict__ tok, int C, int F,
                                      int H, int W, int pt, int ph, int pw) {
  pdl_wait();
  const int Hp = H / ph, Wp = W / pw;
  const int P = C * pt * ph * pw;
  const int64_t total = (int64_t)(F / pt) * Hp * Wp * P;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
    const int64_t n = i / P;
    int p = (int)(i % P);
    const int p0 = p;
    const int f = (int)(n / ((int64_t)Hp * Wp)), h = (int)((n / Wp) % Hp), w = (int)(n % Wp);
    const int dw = p % pw; p /= pw;
    const int dh = p % ph; p /= ph;
    const int dt = p % pt; p /= pt;
    const int c = p;
    const int64_t src = (((int64_t)c * F + (f * pt + dt)) * H + (h * ph + dh)) * W + (w * pw + dw);
    if (!ACID_IN_BOUNDS(kSitePatchify, src, (int64_t)C * F * H * W) ||
        !ACID_IN_BOUNDS(kSitePatchify, n * 2 * P + P + p0, total * 2))
      continue;
    const float x = lat[src];
    const __nv_bfloat16 hi = __float2bfloat16_rn(x);
    tok[n * 2 * P + p0] = hi;
    tok[n * 2 * P + P + p0] = __float2bfloat16_rn(x - __bfloat162float(hi));
  }
}

__global__ void unpatchify_euler_kernel(const float* __restrict__ vtok, float* __restrict__ vout, float* lat, int C,
                                        int F, int H, int W, int pt, int ph, int pw, float dsig) {
  pdl_wait();
  const int Hp = H / ph, Wp = W / pw;
  const int P = C * pt * ph * pw;
  const int64_t total = (int64_t)C * F * H * W;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
    const int w = (int)(i % W);
    const int h = (int)((i / W) % H);
    const int f = (int)((i / ((int64_t)W * H)) % F);
    const int c = (int)(i / ((int64_t)W * H * F));
    const int64_t n = ((int64_t)(f / pt) * Hp + h / ph) * Wp + w / pw;
    const int p = ((c * pt + f % pt) * ph + h % ph) * pw + w % pw;
    if (!ACID_IN_BOUNDS(kSiteUnpatchify, n * P + p, (int64_t)(F / pt) * Hp * Wp * P)) continue;
    const float v = vtok[n * P + p];
    if (vout) vout[i] = v;
    if (lat) lat[i] = fmaf(dsig, v, lat[i]);
  }
}

__global__ void euler_kernel(float* lat, const float* __restrict__ v, int64_t n, float dsig) {
  pdl_wait();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) lat[i] = fmaf(dsig, v[i], lat[i]);
}

// Classifier-free guidance and the Euler step: x += dsig * (v_u + g (v_c - v_u)).
__global__ void guided_euler_kernel(float* lat, const float* __restrict__ vc, const float* __restrict__ vu, int64_t n,
                                    float g, float dsig) {
  pdl_wait();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const float u = vu[i];
    lat[i] = fmaf(dsig, fmaf(g, vc[i] - u, u), lat[i]);
  }
}

// The same with dsigma read from device memory (graph-launched loops).
__global__ void guided_euler_sig_kernel(float* lat, const float* __restrict__ vc, const float* __restrict__ vu,
                                        int64_t n, float g, const double* sig, const int* step) {
  pdl_wait();
  const int i0 = *step;
  const float dsig = (float)(sig[i0 + 1] - sig[i0]);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const float u = vu[i];
    lat[i] = fmaf(dsig, fmaf(g, vc[i] - u, u), lat[i]);
  }
}

// dsigma = sigma[step + 1] - sigma[step] with the step index read from device memory
__global__ void euler_sig_kernel(float* lat, const float* __restrict__ v, int64_t n, const double* sig,
                                 const int* step) {
  pdl_wait();
  const int i0 = *step;
  const float dsig = (float)(sig[i0 + 1] - sig[i0]);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) lat[i] = fmaf(dsig, v[i], lat[i]);
}

int grid_for(int64_t work, int per_block = kThreads, int cap = 152 * 16) {
  int64_t g = (work + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

}  // namespace

ACID_DEVICE_FLAG_READER(take_device_error_elementwise)
ACID_BOUNDS_READER(take_bounds_elementwise)

// =========================================================================
// host launchers
// =========================================================================

size_t drift_workspace_bytes(int64_t) { return sizeof(double2) * kDriftMaxBlocks + 64; }

acid_status drift_launch(int dtype, const void* prev, const void* cur, const void* resid, void* out, int64_t n,
                         double* d_result, void* workspace, size_t ws_bytes, cudaStream_t s, double* rel_out,
                         double* sums_out) {
  ACID_REQUIRE(ws_bytes >= sizeof(double2) * kDriftMaxBlocks, ACID_ERR_WORKSPACE, "drift: workspace too small");
  double2* parts = static_cast<double2*>(workspace);
  const int V = dtype == ACID_BF16 ? 8 : 4;
  const int64_t nvec = n / V;
  int grid = (int)std::min<int64_t>(kDriftMaxBlocks, std::max<int64_t>(1, (nvec + kThreads - 1) / kThreads));
  const double esz = dtype == ACID_BF16 ? 2.0 : 4.0;
  ProfScope prof(PROF_DRIFT, (double)n * esz * (resid ? 4.0 : 2.0), s);  // algorithmic bytes
  if (dtype == ACID_BF16) {
    using T = __nv_bfloat16;
    if (resid)
      launch_pdl(drift_partials_kernel<T, true>, grid, kThreads, 0, s, (const T*)prev, (const T*)cur, (const T*)resid,
                 (T*)out, n, parts);
    else
      launch_pdl(drift_partials_kernel<T, false>, grid, kThreads, 0, s, (const T*)prev, (const T*)cur, nullptr, nullptr,
                 n, parts);
  } else {
    if (resid)
      launch_pdl(drift_partials_kernel<float, true>, grid, kThreads, 0, s, (const float*)prev, (const float*)cur,
                 (const float*)resid, (float*)out, n, parts);
    else
      launch_pdl(drift_partials_kernel<float, false>, grid, kThreads, 0, s, (const float*)prev, (const float*)cur,
                 nullptr, nullptr, n, parts);
  }
  ACID_CHECK_LAUNCH();
  launch_pdl(drift_final_kernel, 1, kThreads, 0, s, parts, grid, d_result, rel_out, sums_out);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

acid_status add_same(int dtype, const void* a, const void* b, void* out, int64_t n, cudaStream_t s) {
  const int V = dtype == ACID_BF16 ? 8 : 4;
  const int grid = grid_for(n / V + 1, kThreads, 152 * 8);
  if (dtype == ACID_BF16)
    launch_pdl(add_vec_kernel<__nv_bfloat16>, grid, kThreads, 0, s, (const __nv_bfloat16*)a, (const __nv_bfloat16*)b,
               (__nv_bfloat16*)out, n);
  else
    launch_pdl(add_vec_kernel<float>, grid, kThreads, 0, s, (const float*)a, (const float*)b, (float*)out, n);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

acid_status add_mixed(int ad, const void* a, int bd, const void* b, int od, void* out, int64_t n, float bs,
                      cudaStream_t s) {
  using H = __nv_bfloat16;
  const bool vec = aligned(a, 16) && aligned(b, 16) && aligned(out, 16);
  const int grid = vec ? grid_for(n / 8 + 1, kThreads, 152 * 8) : grid_for(n);
#define ACID_ADD(TA, TB, TO)                                                                                     \
  launch_pdl(!vec         ? add_mixed_kernel<TA, TB, TO>                                                         \
             : bs == 0.0f ? add_mixed8_kernel<TA, TB, TO, false>                                                 \
                          : add_mixed8_kernel<TA, TB, TO, true>,                                                 \
             grid, kThreads, 0, s, (const TA*)a, (const TB*)b, (TO*)out, n, bs)
  const int key = ad * 4 + bd * 2 + od;  // ACID_BF16 = 0, ACID_FP32 = 1
  switch (key) {
    case 0: ACID_ADD(H, H, H); break;
    case 1: ACID_ADD(H, H, float); break;
    case 2: ACID_ADD(H, float, H); break;
    case 3: ACID_ADD(H, float, float); break;
    case 4: ACID_ADD(float, H, H); break;
    case 5: ACID_ADD(float, H, float); break;
    case 6: ACID_ADD(float, float, H); break;
    default: ACID_ADD(float, float, float); break;
  }
#undef ACID_ADD
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

template <typename Tin, typename Tout, int NV, int MODE>
acid_status launch_ln_rows(const LnArgs& a, cudaStream_t s) {
  constexpr int64_t per_block = kLnThreads / 32;
  const unsigned grid = (unsigned)((a.rows + per_block - 1) / per_block);
  if (a.d == 128 * NV)
    launch_pdl(ln_mod_rows_kernel<Tin, Tout, NV, true, MODE>, grid, kLnThreads, 0, s, a);
  else
    launch_pdl(ln_mod_rows_kernel<Tin, Tout, NV, false, MODE>, grid, kLnThreads, 0, s, a);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

template <typename Tin, typename Tout, int WPR, int NQ, bool FULL, int MODE>
acid_status launch_ln_team(const LnArgs& a, cudaStream_t s) {
  constexpr size_t kSmemMax = 216 * 1024 / kLnCtas<WPR>;
  static PerContext allowed;
  ACID_TRY(allow_smem(allowed, ln_mod_team_kernel<Tin, Tout, WPR, NQ, FULL, MODE>, kSmemMax));
  const size_t row = (size_t)a.d * (MODE == kLnPlain ? sizeof(Tin) : MODE == kLnReuse ? 8 : sizeof(Tin) + 4);
  // Two rows ahead keep HBM busy and its reads in order (bf16, 50000 x 3072: 93 us,
  // 109 with four); rows that largely stay in L2 are latency's, which four cover
  // (16000 x 1920: 19.5 us, 21.4 with two; the line lies between 154 and 200 MB).
  const double bytes = (double)a.rows * a.d * (sizeof(Tin) + sizeof(Tout));
  const int stages = row <= 6144 && bytes < 160e6 ? kLnMaxStages : 2;
  const unsigned grid = (unsigned)std::min<int64_t>(a.rows, (int64_t)num_sms() * kLnCtas<WPR>);
  launch_pdl(ln_mod_team_kernel<Tin, Tout, WPR, NQ, FULL, MODE>, grid, 32 * WPR, stages * row, s, a, stages);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

template <typename Tin, typename Tout, int WPR, int NQ, int MODE>
acid_status launch_ln_team(const LnArgs& a, cudaStream_t s) {
  return a.d == 128 * WPR * NQ ? launch_ln_team<Tin, Tout, WPR, NQ, true, MODE>(a, s)
                               : launch_ln_team<Tin, Tout, WPR, NQ, false, MODE>(a, s);
}

// Warps and quads per lane sized to the row.
template <typename Tin, typename Tout, int MODE>
acid_status ln_mod_types(const LnArgs& a, cudaStream_t s) {
  if (a.d <= 512) return launch_ln_rows<Tin, Tout, 4, MODE>(a, s);
  if (a.d <= 1536) return launch_ln_team<Tin, Tout, 2, 6, MODE>(a, s);
  if (a.d <= 1920) return launch_ln_team<Tin, Tout, 3, 5, MODE>(a, s);
  return launch_ln_team<Tin, Tout, 4, 6, MODE>(a, s);
}

acid_status ln_mod(int in_dtype, const void* x, int out_dtype, void* y, int64_t rows, int d, const float* shv,
                   const float* scv, const float* sht, const float* sct, int64_t split, float eps, cudaStream_t s) {
  using H = __nv_bfloat16;
  ACID_REQUIRE(d % 8 == 0 && d <= 3072, ACID_ERR_UNSUPPORTED, "ln_mod: d must be a multiple of 8, <= 3072");
  if (rows == 0) return ACID_OK;
  ACID_REQUIRE(aligned(shv, 16) && aligned(scv, 16) && aligned(sht, 16) && aligned(sct, 16), ACID_ERR_UNSUPPORTED,
               "ln_mod: shift and scale must be 16-byte aligned");
  const bool two = scv != nullptr && sht != nullptr && split > 0 && (sht != shv || sct != scv);
  const LnArgs a{x, y, nullptr, nullptr, rows, split, d, scv == nullptr ? 0 : two ? 2 : 1, shv, scv, sht, sct, eps};
  if (in_dtype == ACID_BF16 && out_dtype == ACID_BF16) return ln_mod_types<H, H, kLnPlain>(a, s);
  if (in_dtype == ACID_BF16) return ln_mod_types<H, float, kLnPlain>(a, s);
  if (out_dtype == ACID_BF16) return ln_mod_types<float, H, kLnPlain>(a, s);
  return ln_mod_types<float, float, kLnPlain>(a, s);
}

acid_status ln_mod_cached(int dtype, bool reuse, const void* x, const float* h, float* r, void* y, int64_t rows, int d,
                          const float* sh, const float* sc, float eps, cudaStream_t s) {
  using H = __nv_bfloat16;
  ACID_REQUIRE(d % 8 == 0 && d <= 3072, ACID_ERR_UNSUPPORTED, "ln_mod: d must be a multiple of 8, <= 3072");
  if (rows == 0) return ACID_OK;
  const LnArgs a{x, y, h, r, rows, 0, d, 1, sh, sc, nullptr, nullptr, eps};
  if (dtype == ACID_BF16) return reuse ? ln_mod_types<H, H, kLnReuse>(a, s) : ln_mod_types<H, H, kLnResid>(a, s);
  return reuse ? ln_mod_types<float, float, kLnReuse>(a, s) : ln_mod_types<float, float, kLnResid>(a, s);
}

template <int NV4, int WPR>
acid_status launch_temni_drift(const float* h_cur, const float* h_prev, const float* mod_cur, const float* mod_prev,
                               const int* step_dev, int step_host, int64_t rows, int d, float eps, double2* parts,
                               unsigned int* done, double* result, cudaStream_t s, int* grid_out) {
  constexpr int kSmemMax = 225 * 1024;  // dynamic shared memory, below the 227 KB limit less the static part
  static PerContext allowed;
  ACID_TRY(allow_smem(allowed, temni_drift_kernel<NV4, WPR>, kSmemMax));
  // groups per CTA: as many two-stage rings (8 d bytes per stage) as fit
  // beside the staged modulation vectors (16 d bytes), within the group and
  // warp limits
  const size_t ring_per_group = (size_t)kTemniStages * 8 * d + kTemniStages * sizeof(uint64_t);
  const int groups = (int)std::max<size_t>(1, std::min<size_t>(std::min(kTemniMaxGroups, kTemniMaxWarps / WPR),
                                                               (kSmemMax - 16 * (size_t)d) / ring_per_group));
  const size_t smem = 16 * (size_t)d + groups * ring_per_group;
  const int grid = (int)std::min<int64_t>(std::min<int64_t>(kDriftMaxBlocks, (int64_t)num_sms()),
                                          std::max<int64_t>(1, (rows + groups - 1) / groups));
  launch_pdl(temni_drift_kernel<NV4, WPR>, grid, 32 * WPR * groups, smem, s, h_cur, h_prev, step_dev, step_host, rows,
             d, mod_cur, mod_cur + d, mod_prev, mod_prev + d, eps, parts, done, result);
  ACID_CHECK_LAUNCH();
  *grid_out = grid;
  return ACID_OK;
}

acid_status temni_drift(const float* h_cur, const float* h_prev, const float* mod_cur, const float* mod_prev,
                        const int* step_dev, int step_host, int64_t rows, int d, float eps, double* d_result,
                        void* workspace, size_t ws_bytes, cudaStream_t s, unsigned int* done, double* rel_out,
                        double* sums_out) {
  ACID_REQUIRE(d % 8 == 0 && d <= 3072, ACID_ERR_UNSUPPORTED, "temni_drift: d must be a multiple of 8, <= 3072");
  ACID_REQUIRE(ws_bytes >= sizeof(double2) * kDriftMaxBlocks, ACID_ERR_WORKSPACE, "temni_drift: workspace too small");
  ACID_REQUIRE(aligned(h_cur, 16) && aligned(h_prev, 16) && aligned(mod_cur, 16) && aligned(mod_prev, 16),
               ACID_ERR_UNSUPPORTED, "temni_drift: inputs must be 16-byte aligned");
  double2* parts = static_cast<double2*>(workspace);
  ProfScope prof(PROF_DRIFT, (double)rows * d * 8.0, s);  // read both steps' H_in (fp32)
  int grid = 1;
  auto run = [&](auto nv4, auto wpr) {
    return launch_temni_drift<decltype(nv4)::value, decltype(wpr)::value>(
        h_cur, h_prev, mod_cur, mod_prev, step_dev, step_host, rows, d, eps, parts, done, d_result, s, &grid);
  };
  using std::integral_constant;
  if (d <= 512)
    ACID_TRY(run(integral_constant<int, 4>{}, integral_constant<int, 1>{}));
  else if (d <= 1536)
    // 66.5 us at 32760 x 1536; two warps a row: 68.8
    ACID_TRY(run(integral_constant<int, 12>{}, integral_constant<int, 1>{}));
  else if (d <= 2048)
    ACID_TRY(run(integral_constant<int, 4>{}, integral_constant<int, 4>{}));
  else
    ACID_TRY(run(integral_constant<int, 6>{}, integral_constant<int, 4>{}));
  if (done == nullptr) {
    launch_pdl(drift_final_kernel, 1, kThreads, 0, s, parts, grid, d_result, rel_out, sums_out);
    ACID_CHECK_LAUNCH();
  }
  return ACID_OK;
}

namespace {
template <typename TW>
acid_status launch_gemv(const GemvMat& m0, const GemvMat& m1, const float* x, int k, bool silu_input, cudaStream_t s) {
  const int total = m0.n_out + m1.n_out;
  const size_t smem = sizeof(float) * k;
  // four rows per warp, on as many CTAs as are resident, once every SM gets two
  constexpr int kWarps = kThreads / 32;
  const int sms = num_sms();
  auto grid = [&](int rows) { return std::min((total + kWarps * rows - 1) / (kWarps * rows), sms * 3); };
  if (total >= sms * 2 * kWarps * 4)
    launch_pdl(gemv_kernel<TW, 4>, grid(4), kThreads, smem, s, m0, m1, x, k, silu_input);
  else if (total >= sms * 2 * kWarps * 2)
    launch_pdl(gemv_kernel<TW, 2>, grid(2), kThreads, smem, s, m0, m1, x, k, silu_input);
  else
    launch_pdl(gemv_kernel<TW, 1>, grid(1), kThreads, smem, s, m0, m1, x, k, silu_input);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}
}  // namespace

acid_status gemv2(int w_dtype, const void* W, const float* b, float* y, int n_out, const void* W2, const float* b2,
                  float* y2, int n_out2, const float* x, int k, bool silu_input, cudaStream_t s) {
  ACID_REQUIRE(k % 8 == 0 && k <= 16384, ACID_ERR_UNSUPPORTED, "gemv: k must be a multiple of 8, <= 16384");
  ACID_REQUIRE(aligned(W, 16) && aligned(W2, 16), ACID_ERR_UNSUPPORTED,
               "gemv: time and modulation weights must be 16-byte aligned");
  const GemvMat m0{W, b, y, n_out}, m1{W2, b2, y2, n_out2};
  return w_dtype == ACID_BF16 ? launch_gemv<__nv_bfloat16>(m0, m1, x, k, silu_input, s)
                              : launch_gemv<float>(m0, m1, x, k, silu_input, s);
}

acid_status gemv(int w_dtype, const void* W, const float* b, const float* x, float* y, int n_out, int k,
                 bool silu_input, cudaStream_t s) {
  return gemv2(w_dtype, W, b, y, n_out, nullptr, nullptr, nullptr, 0, x, k, silu_input, s);
}

acid_status timestep_sinusoid(float* out, double t, int dim, cudaStream_t s) {
  const int half = dim / 2;
  launch_pdl(sinusoid_kernel, dim3((half + kTableThreads - 1) / kTableThreads, 2), kTableThreads, 0, s, out, t, half);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

RopeTable rope_layout(int grid_f, int grid_h, int grid_w, int head_dim) {
  RopeTable t;
  const int dh = 2 * (head_dim / 6);
  const int dt = head_dim - 2 * dh;
  t.grid_f = grid_f; t.grid_h = grid_h; t.grid_w = grid_w;
  t.pairs_t = dt / 2; t.pairs_h = dh / 2; t.pairs_w = dh / 2;
  if (grid_h > 0 && grid_w > 0) {
    t.inv_hw = 1.0f / (float)(grid_h * grid_w);
    t.inv_w = 1.0f / (float)grid_w;
  }
  return t;
}

acid_status rope_build(RopeTable& t, float2* storage, float theta, cudaStream_t s) {
  t.table = storage;
  const int64_t total = t.elems();
  if (total == 0) return ACID_OK;
  const dim3 grid((unsigned)((total + kTableThreads - 1) / kTableThreads), 2);
  launch_pdl(rope_table_kernel, grid, kTableThreads, 0, s, storage, t.grid_f, t.grid_h, t.grid_w, t.pairs_t, t.pairs_h,
             t.pairs_w, (double)theta);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

namespace {
// grid and shared memory of the tile kernels; false if the patch is too long
// (or the grid too tall) for them
bool patch_tiles(const PatchGeo& g, dim3* grid, size_t* smem) {
  const int P = g.C * g.pt * g.ph * g.pw;
  const int Wp = g.W / g.pw, Hp = g.H / g.ph, Fp = g.F / g.pt;
  if (P > kPatchMaxP || Hp > 65535 || Fp > 65535) return false;
  *grid = dim3((unsigned)((Wp + kPatchTile - 1) / kPatchTile), (unsigned)Hp, (unsigned)Fp);
  *smem = sizeof(float) * kPatchTile * (P + 1);
  return true;
}
}  // namespace

acid_status patchify(const float* latent, float* tokens, int C, int F, int H, int W, int pt, int ph, int pw,
                     cudaStream_t s) {
  const PatchGeo g{C, F, H, W, pt, ph, pw};
  dim3 grid;
  size_t smem;
  if (patch_tiles(g, &grid, &smem))
    launch_pdl(patchify_tile_kernel<false>, grid, kThreads, smem, s, latent, (void*)tokens, g);
  else
    launch_pdl(patchify_kernel, grid_for((int64_t)C * F * H * W), kThreads, 0, s, latent, tokens, C, F, H, W, pt, ph,
               pw);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

acid_status patchify_split(const float* latent, void* tokens, int C, int F, int H, int W, int pt, int ph, int pw,
                           cudaStream_t s) {
  const PatchGeo g{C, F, H, W, pt, ph, pw};
  dim3 grid;
  size_t smem;
  if (patch_tiles(g, &grid, &smem))
    launch_pdl(patchify_tile_kernel<true>, grid, kThreads, smem, s, latent, tokens, g);
  else
    launch_pdl(patchify_split_kernel, grid_for((int64_t)C * F * H * W), kThreads, 0, s, latent, (__nv_bfloat16*)tokens,
               C, F, H, W, pt, ph, pw);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

acid_status unpatchify_euler(const float* vtok, float* v_out, float* latent, int C, int F, int H, int W, int pt,
                             int ph, int pw, float dsigma, cudaStream_t s) {
  const PatchGeo g{C, F, H, W, pt, ph, pw};
  dim3 grid;
  size_t smem;
  if (patch_tiles(g, &grid, &smem))
    launch_pdl(unpatchify_tile_kernel, grid, kThreads, smem, s, vtok, v_out, latent, g, dsigma);
  else
    launch_pdl(unpatchify_euler_kernel, grid_for((int64_t)C * F * H * W), kThreads, 0, s, vtok, v_out, latent, C, F, H,
               W, pt, ph, pw, dsigma);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

acid_status euler_update(float* latent, const float* v, int64_t n, float dsigma, cudaStream_t s) {
  launch_pdl(euler_kernel, grid_for(n), kThreads, 0, s, latent, v, n, dsigma);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

acid_status guided_euler_update(float* latent, const float* v_cond, const float* v_uncond, int64_t n, float scale,
                               float dsigma, cudaStream_t s) {
  launch_pdl(guided_euler_kernel, grid_for(n), kThreads, 0, s, latent, v_cond, v_uncond, n, scale, dsigma);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

acid_status guided_euler_update_sig(float* latent, const float* v_cond, const float* v_uncond, int64_t n, float scale,
                                   const double* sig, const int* step, cudaStream_t s) {
  launch_pdl(guided_euler_sig_kernel, grid_for(n), kThreads, 0, s, latent, v_cond, v_uncond, n, scale, sig, step);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

acid_status euler_update_sig(float* latent, const float* v, int64_t n, const double* sig, const int* step,
                             cudaStream_t s) {
  launch_pdl(euler_sig_kernel, grid_for(n), kThreads, 0, s, latent, v, n, sig, step);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

acid_status timestep_sinusoid_sig(float* out, const double* sig, const int* step, int dim, cudaStream_t s) {
  const int half = dim / 2;
  launch_pdl(sinusoid_sig_kernel, dim3((half + kTableThreads - 1) / kTableThreads, 2), kTableThreads, 0, s, out, sig,
             step, half);
  ACID_CHECK_LAUNCH();
  return ACID_OK;
}

}  // namespace acid
