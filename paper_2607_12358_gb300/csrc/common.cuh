// Shared device helpers: bf16 packing, bounded mbarrier waits, TMA and
// tcgen05 (5th-generation tensor core) wrappers written as inline PTX for
// sm_103a, and the host-side status plumbing of the C ABI.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <string>
#include <utility>

#include "acid.h"

namespace acid {

// ---------------------------------------------------------------------------
// Host-side status handling
// ---------------------------------------------------------------------------
void set_error(const std::string& msg);
void clear_error();

#define ACID_REQUIRE(cond, code, msg)          \
  do {                                         \
    if (!(cond)) {                             \
      ::acid::set_error(msg);                  \
      return (code);                           \
    }                                          \
  } while (0)

#define ACID_CUDA(call)                                                        \
  do {                                                                         \
    cudaError_t e_ = (call);                                                   \
    if (e_ != cudaSuccess) {                                                   \
      ::acid::set_error(std::string(#call) + ": " + cudaGetErrorString(e_));   \
      return ACID_ERR_CUDA;                                                    \
    }                                                                          \
  } while (0)

// Id of the calling thread's CUDA context, never given to another one; 0 if it
// has none yet (or the driver cannot tell).
unsigned long long context_id();

// A number in 1 .. 65535 that is asked for once in each CUDA context (so for each
// device, and again after a device reset): the kernels' shared memory opt-in,
// which belongs to a device, and what was counted there.  Safe from several
// threads: two that ask at once both call make, which has to allow that.  A
// lookup takes 6 ns; cudaFuncSetAttribute at each launch would take 200.
class PerContext {
 public:
  // make(&value) forms the number; a status other than ACID_OK is passed on and nothing is kept.
  template <typename F>
  acid_status get(int* value, F make) {
    unsigned long long id = context_id();
    const unsigned long long kept = slot_[id % kSlots].load(std::memory_order_acquire);
    if (id != 0 && kept >> 16 == id) {
      *value = (int)(kept & 0xffff);
      return ACID_OK;
    }
    const acid_status st = make(value);
    if (st != ACID_OK) return st;
    id = context_id();  // make may have been this thread's first use of the device
    if (id != 0 && *value > 0 && *value < 65536)
      slot_[id % kSlots].store(id << 16 | (unsigned long long)*value, std::memory_order_release);
    return ACID_OK;
  }

 private:
  static constexpr int kSlots = 16;  // contexts that share a slot ask again
  std::atomic<unsigned long long> slot_[kSlots] = {};
};

// Raises a kernel's dynamic shared memory limit where it has not been raised yet.
template <typename K>
acid_status allow_smem(PerContext& done, K kernel, size_t bytes) {
  int yes;
  return done.get(&yes, [&](int* v) {
    *v = 1;
    ACID_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    return ACID_OK;
  });
}

// SMs of the current device.
int num_sms();

// Counts every kernel launch of the library (acid_launch_count) and checks it.
void count_launch();
#define ACID_CHECK_LAUNCH()   \
  do {                        \
    ::acid::count_launch();   \
    ACID_CUDA(cudaGetLastError()); \
  } while (0)

// Launches a kernel that may start while the kernel before it on the stream is
// still draining (programmatic dependent launch): its launch and set-up
// overlap that kernel's tail.  Every kernel launched this way calls pdl_wait
// before its first access to global memory, which returns once the kernel
// before has completed and its writes are visible, so the stream's order of
// effects is kept, link by link.
//   Kernels leave the moment their successor may start to the default, the end
// of their CTAs.  Allowed earlier, the successor's CTAs pile up on the few SMs
// that the running kernel leaves free: a 128-CTA fp32 GEMM in a chain ran
// 17.5 us instead of 9.2, the toy generation 1187 us instead of 1018.
template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}
// Records CUDA events around one launch on its stream while profiling is on
// (acid_profile_enable); `work` is the launch's algorithmic FLOPs or bytes.
enum ProfKind { PROF_ATTENTION = 0, PROF_LINEAR = 1, PROF_DRIFT = 2, PROF_KINDS = 3 };
class ProfScope {
 public:
  ProfScope(int kind, double work, cudaStream_t s);
  ~ProfScope();

 private:
  int slot_ = -1;
  cudaStream_t s_;
};

#define ACID_TRY(expr)                 \
  do {                                 \
    acid_status s_ = (expr);           \
    if (s_ != ACID_OK) return s_;      \
  } while (0)

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Device flag raised by a bounded wait that ran out (see acid_check_device_error).
// One copy per translation unit (no relocatable device code); each unit that
// waits exports a reader through ACID_DEVICE_FLAG_READER.  A unit that defines
// ACID_UNIT_WITHOUT_WAITS has neither the flag nor the functions that raise it.
#ifndef ACID_UNIT_WITHOUT_WAITS
static __device__ unsigned int g_device_error = 0;

#define ACID_DEVICE_FLAG_READER(fname)                                              \
  unsigned int fname() {                                                           \
    unsigned int v = 0, z = 0;                                                     \
    if (cudaMemcpyFromSymbol(&v, g_device_error, sizeof(v)) != cudaSuccess) return 2; \
    if (v) cudaMemcpyToSymbol(g_device_error, &z, sizeof(z));                      \
    return v;                                                                      \
  }
#endif

// Debug builds (compiled with ACID_BOUNDS_CHECK, libacid_gb300_debug.so)
// check the global-memory index of the kernels' hand-computed accesses
// against the extent the host passed: ACID_IN_BOUNDS(site, i, n) is true for
// 0 <= i < n; otherwise it records the translation unit's first violation
// {site, index, extent} and returns false, and the caller skips the access.
// Release builds compile every check to `true`.  Accesses made by the TMA
// engine are bounded by their tensor maps and are not checked here.
enum BoundsSite : int {
  kSiteDrift = 1, kSiteAdd = 2, kSiteLayerNorm = 3, kSiteTemni = 4, kSitePatchify = 5, kSiteUnpatchify = 6,
  kSiteGemv = 7, kSiteGemmResidual = 8, kSiteGemmStore = 9, kSiteGemmRope = 10, kSiteGemmF32 = 11,
  kSiteAttnMerge = 12, kSiteAttnF32 = 13, kSiteSelftest = 99
};
struct BoundsRecord {
  long long site, index, extent;
};
static __device__ BoundsRecord g_bounds = {0, 0, 0};
#ifdef ACID_BOUNDS_CHECK
static __device__ __noinline__ bool bounds_fail(int site, long long i, long long n) {
  if (atomicCAS(reinterpret_cast<unsigned long long*>(&g_bounds.site), 0ull, (unsigned long long)site) == 0ull) {
    g_bounds.index = i;
    g_bounds.extent = n;
  }
  return false;
}
#define ACID_IN_BOUNDS(site, i, n)                                                   \
  (((long long)(i) >= 0 && (long long)(i) < (long long)(n)) ? true                   \
                                                           : ::acid::bounds_fail((site), (long long)(i), (long long)(n)))
constexpr bool kBoundsChecked = true;
#else
#define ACID_IN_BOUNDS(site, i, n) true
constexpr bool kBoundsChecked = false;
#endif
// Host reader of the translation unit's record (cleared after reading).
#define ACID_BOUNDS_READER(fname)                                                    \
  BoundsRecord fname() {                                                             \
    BoundsRecord r{0, 0, 0}, z{0, 0, 0};                                             \
    if (cudaMemcpyFromSymbol(&r, g_bounds, sizeof(r)) != cudaSuccess) r.site = -1;   \
    else if (r.site) cudaMemcpyToSymbol(g_bounds, &z, sizeof(z));                    \
    return r;                                                                        \
  }

// ---------------------------------------------------------------------------
// Programmatic dependent launch (see launch_pdl)
// ---------------------------------------------------------------------------
// Waits until the kernel before this one has completed.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Numeric helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}

template <typename T> struct io;
template <> struct io<float> {
  static __device__ __forceinline__ float ld(const float* p) { return *p; }
  static __device__ __forceinline__ void st(float* p, float v) { *p = v; }
};
template <> struct io<__nv_bfloat16> {
  static __device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  static __device__ __forceinline__ void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
};

// 8 consecutive values <-> fp32 registers (16 bytes of bf16, 32 bytes of fp32)
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float* v) {
  uint4 u = *reinterpret_cast<const uint4*>(p);
  v[0] = bf16_lo(u.x); v[1] = bf16_hi(u.x); v[2] = bf16_lo(u.y); v[3] = bf16_hi(u.y);
  v[4] = bf16_lo(u.z); v[5] = bf16_hi(u.z); v[6] = bf16_lo(u.w); v[7] = bf16_hi(u.w);
}
__device__ __forceinline__ void load8(const float* p, float* v) {
  float4 a = *reinterpret_cast<const float4*>(p);
  float4 b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float* v) {
  uint4 u;
  u.x = pack_bf16(v[0], v[1]); u.y = pack_bf16(v[2], v[3]);
  u.z = pack_bf16(v[4], v[5]); u.w = pack_bf16(v[6], v[7]);
  *reinterpret_cast<uint4*>(p) = u;
}
__device__ __forceinline__ void store8(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}

// GELU, tanh form: 0.5 x (1 + tanh(sqrt(2/pi) (x + 0.044715 x^3))).
// The bf16 path uses the hardware tanh approximation (tanh.approx.f32,
// relative error about 2^-11, below bf16 output rounding); the fp32 path
// calls tanhf.
__device__ __forceinline__ float tanh_fast(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
template <bool kFast>
__device__ __forceinline__ float gelu_tanh(float x) {
  const float k0 = 0.7978845608028654f;  // sqrt(2/pi)
  const float u = k0 * fmaf(0.044715f * x, x * x, x);
  const float t = kFast ? tanh_fast(u) : tanhf(u);
  return 0.5f * x * (1.0f + t);
}

__device__ __forceinline__ float silu(float x) { return x / (1.0f + expf(-x)); }

// Packed fp32 pair arithmetic (one instruction for two lanes of work).
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---------------------------------------------------------------------------
// mbarrier (bounded waits)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// About 4 s at 2 GHz: far above any legitimate wait in these kernels.
constexpr long long kWaitLimitCycles = 8000000000LL;

#ifndef ACID_UNIT_WITHOUT_WAITS
// Returns false (and raises the device flag) if the phase did not complete
// within `limit` SM clocks.  Callers stop their role's loop on false.
__device__ __forceinline__ bool mbar_wait_limit(uint64_t* bar, uint32_t parity, long long limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    #pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (clock64() - t0 > limit) {
      atomicExch(&g_device_error, 1u);
      return false;
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  return mbar_wait_limit(bar, parity, kWaitLimitCycles);
}

// The same by every lane of a warp: one warp-uniform answer.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity));
}
#endif
// Warp index as a value the compiler knows to be the same in all lanes.
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }
// True in one lane of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(p));
  return p != 0;
}

// ---------------------------------------------------------------------------
// cp.async and named barriers (the FP32-pipe kernels)
// ---------------------------------------------------------------------------
// n bytes (4 or 16) from global to shared memory; zeros when !valid.
template <int N>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool valid) {
  const int sz = valid ? N : 0;
  if constexpr (N == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(sz) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(sz) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// Barrier `id` (1..15) among `threads` threads of the CTA.
__device__ __forceinline__ void group_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// The same, and whether `vote` is true in all of them: one answer for the whole
// group, which belongs to this barrier.  (A flag in shared memory read behind
// the barrier can already hold what a faster warp found in its next round.)
__device__ __forceinline__ bool group_all(int id, int threads, bool vote) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred v, a;\n\t"
      "setp.ne.u32 v, %3, 0;\n\t"
      "bar.red.and.pred a, %1, %2, v;\n\t"
      "selp.u32 %0, 1, 0, a;\n\t}"
      : "=r"(r)
      : "r"(id), "r"(threads), "r"((uint32_t)vote)
      : "memory");
  return r != 0;
}

// ---------------------------------------------------------------------------
// TMA (cp.async.bulk.tensor), 2D tiles, 128-byte swizzle
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
// x: innermost (column) element coordinate, must be a multiple of 8 (16 bytes of bf16)
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::
          "r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// Tensor store of one 2D box from shared memory, tracked in the issuing
// thread's bulk async-groups.  x as for tma_load_2d; x, y >= 0 (the box is
// clipped at the far edges of the tensor).  The writes to src must be made
// visible to the async proxy first (fence_proxy_async_smem by every writer).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(src)), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// at most N of this thread's bulk groups still reading their shared-memory source
template <int N>
__device__ __forceinline__ void bulk_wait_group_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
// at most N of this thread's bulk groups not yet complete (writes performed)
template <int N>
__device__ __forceinline__ void bulk_wait_group() {
  asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------------------
// tcgen05: TMEM allocation, MMA, commit, TMEM <-> registers
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor for a 128-byte-swizzled operand tile whose
// 8-row groups are `sbo` bytes apart and whose 64-element (128-byte) column
// chunks are `lbo` bytes apart (lbo matters only for MN-major operands).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version for tcgen05
  d |= (uint64_t)2 << 61;  // 128-byte swizzle
  return d;
}

// Instruction descriptor of kind::f16 with bf16 A/B, fp32 accumulator.
// a_mn / b_mn: operand stored MN-major (transposed) instead of K-major.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N, bool a_mn, bool b_mn) {
  return (1u << 4)                      // D format: f32
         | (1u << 7)                    // A format: bf16
         | (1u << 10)                   // B format: bf16
         | ((a_mn ? 1u : 0u) << 15)     // A major
         | ((b_mn ? 1u : 0u) << 16)     // B major
         | ((uint32_t)(N >> 3) << 17)   // N / 8
         | ((uint32_t)(M >> 4) << 24);  // M / 16
}

__device__ __forceinline__ void mma_bf16_ss(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// A operand from tensor memory (M=128 lanes, 16-bit elements packed two per
// 32-bit column, K along columns), B from shared memory.
__device__ __forceinline__ void mma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrives once on `bar` when every tcgen05 operation issued so far by this
// thread has completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

// 32 lanes x 32 columns of 32-bit: thread i of the warp receives lane
// (base lane + i), columns [col, col + 32).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]),
      "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
      "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------------------
// CTA pairs (clusters of two CTAs on two SMs) and the pair-wide tcgen05 forms
// (cta_group::2): one MMA of M = 256 reads A rows 0-127 and B's first half
// from the shared memory of CTA rank 0 and A rows 128-255 and B's second
// half from rank 1 (same offsets), and writes each CTA's 128 accumulator rows
// into that CTA's TMEM.  A kernel uses either these or the cta_group::1 forms
// above for all of its tcgen05 instructions, never both.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Every thread of both CTAs: arrive and wait on the cluster barrier.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address in the cluster's shared window of the variable at the same offset
// as `local` (a shared::cta address) in the shared memory of CTA `rank`.
__device__ __forceinline__ uint32_t mapa_shared(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
// Arrive once on an mbarrier in either CTA of the cluster.  Default (CTA
// scope) semantics: the barriers it is used on hand over tensor memory, whose
// ordering the tcgen05 fences and waits provide; a cluster-scope release would
// also wait for every earlier global store of the thread to be performed.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// try_wait with acquire at cluster scope (arrivals from the peer CTA).
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
#ifndef ACID_UNIT_WITHOUT_WAITS
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    #pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait_cluster(bar, parity)) return true;
    if (clock64() - t0 > kWaitLimitCycles) {
      atomicExch(&g_device_error, 1u);
      return false;
    }
  }
}
#endif
// TMA tile load into this CTA's shared memory whose completion is counted on
// an mbarrier that may live in either CTA of the pair (cluster address).
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* map, uint32_t bar_cluster, int x,
                                                 int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
      "[%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster), "r"(x), "r"(y)
      : "memory");
}
// Pair-wide TMEM allocation: one warp of each CTA of the pair executes it and
// both receive the same column address.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// Pair-wide MMA (issued by one thread of CTA rank 0), operands as above.
__device__ __forceinline__ void mma_bf16_ss_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                 uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives once on the mbarrier at `bar_cluster` (either CTA of the pair) when
// every pair-wide tcgen05 operation issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar_cluster) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar_cluster)
               : "memory");
}
// The same on the mbarrier at this offset (a shared::cta address) in both CTAs
// of the pair, with one instruction.
__device__ __forceinline__ void mma_commit_both(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}

}  // namespace acid
