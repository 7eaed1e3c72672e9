"""CPU checks of what the launchers do on the host: the library's objects linked
against a stand-in CUDA runtime (a few entry points that record their calls or
answer as told, every other one a stub that returns 0), in a child process
each, so that devices, contexts and failing queries can be played through
without a GPU.  Pointers are made up: nothing on the host reads them."""

import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2607_12358_gb300")

RUNTIME = r"""
#include <cudaTypedefs.h>
#include <cuda_runtime_api.h>
#include <cstring>
#include <map>
#include <set>
#include <utility>

static std::set<std::pair<const void*, int>> opted_in;  // (kernel, device)
static cudaError_t last_error = cudaSuccess;
// the translation units' device error flags (g_device_error) by their host address, numbered as they are registered
static std::map<const void*, int>& flags() {
  static std::map<const void*, int> f;
  return f;
}

extern "C" {
// what the stand-in answers; contexts keep their handle over a reset, not their id
int fk_pairs = 76, fk_occupancy_error = 0, fk_device = 0, fk_attribute_error = 0, fk_resets = 0;
// what it was asked
int fk_launches = 0, fk_grid = 0, fk_lookups = 0;
// device of the memory at 0x2......., its type (cudaMemoryType); copies there, and stores by the drift's final kernel
int fk_home = 0, fk_type = cudaMemoryTypeDevice, fk_copies = 0, fk_stores = 0;
#define OUTPUT(p) (((size_t)(p) >> 28) == 2)

// which of the flags is raised; how many there are
int fk_raised = -1, fk_flags = 0;
void __cudaRegisterVar(void**, char* host, char*, const char* name, int, size_t, int, int) {
  if (std::strstr(name, "g_device_error")) flags()[host] = fk_flags++;
}
cudaError_t cudaMemcpyFromSymbol(void* dst, const void* sym, size_t n, size_t, cudaMemcpyKind) {
  std::memset(dst, 0, n);
  const auto f = flags().find(sym);
  if (f != flags().end() && f->second == fk_raised) *(unsigned*)dst = 1;
  return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbol(const void* sym, const void*, size_t, size_t, cudaMemcpyKind) {
  const auto f = flags().find(sym);
  if (f != flags().end() && f->second == fk_raised) fk_raised = -1;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = fk_device; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  *a = {};
  a->type = OUTPUT(p) ? (cudaMemoryType)fk_type : cudaMemoryTypeDevice;
  a->device = OUTPUT(p) ? fk_home : fk_device;
  a->devicePointer = const_cast<void*>(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void*, size_t, cudaMemcpyKind, cudaStream_t) {
  fk_copies += OUTPUT(dst);
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return std::exchange(last_error, cudaSuccess); }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int) {
  if (fk_attribute_error == 0) opted_in.insert({f, fk_device});
  return (cudaError_t)fk_attribute_error;
}

cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = fk_pairs;
  return (cudaError_t)fk_occupancy_error;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int dev) { *v = dev == 0 ? 152 : 100; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  // more than 48 KB of dynamic shared memory has to be asked for on each device
  if (c->dynamicSmemBytes > 48 * 1024 && !opted_in.count({f, fk_device})) return last_error = cudaErrorInvalidValue;
  ++fk_launches;
  fk_grid = (int)c->gridDim.x;
  if (c->gridDim.x == 1 && c->blockDim.x == 256)  // drift_final_kernel(partials, nparts, result, rel_out, sums_out)
    fk_stores += OUTPUT(*(void**)args[3]) + OUTPUT(*(void**)args[4]);
  return cudaSuccess;
}
static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                       const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
static CUresult ctx_id(CUcontext, unsigned long long* id) {
  *id = 2 * fk_resets + fk_device + 1;
  return CUDA_SUCCESS;
}
static CUresult ctx_current(CUcontext* c) { *c = (CUcontext)(size_t)(0x1000 + fk_device); return CUDA_SUCCESS; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = (void*)(size_t)(0x30000000 + 0x10000 * ++fk_lookups);
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** fn, unsigned int, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *fn = !std::strcmp(name, "cuTensorMapEncodeTiled") ? (void*)encode
        : !std::strcmp(name, "cuCtxGetId")           ? (void*)ctx_id
        : !std::strcmp(name, "cuCtxGetCurrent")      ? (void*)ctx_current
                                                      : nullptr;
  *q = *fn ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "stand-in error"; }
}
"""

# lib: the library under test; fk: its runtime's knobs and records; A: the binding's constants
PRELUDE = r"""
import ctypes as C, importlib.util, sys
spec = importlib.util.spec_from_file_location("capi", sys.argv[2])
A = importlib.util.module_from_spec(spec)
spec.loader.exec_module(A)
lib = C.CDLL(sys.argv[1])
for name, (res, args) in A._PROTOS.items():
    getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
rt = C.CDLL(sys.argv[3]) if len(sys.argv) > 3 else None
class Fk:
    def __getattr__(self, n): return C.c_int.in_dll(rt, "fk_" + n).value
    def __setattr__(self, n, v): C.c_int.in_dll(rt, "fk_" + n).value = v
fk = Fk()
p = [0x10000000 + 0x1000000 * i for i in range(16)]  # addresses that nothing reads
def linear(dtype=A.ACID_BF16, M=512, K=1536, N=3072, epi=A.ACID_EPI_BIAS, out_fp32=0):
    res = epi in (A.ACID_EPI_GATED_RES, A.ACID_EPI_RES)
    return lib.acid_linear_forward(dtype, p[0], K, M, K, p[1], None, N, p[2], N, epi,
                                   p[4] if epi == A.ACID_EPI_GATED_RES else None, p[3] if res else None,
                                   N if res else 0, out_fp32, None)
def attention(dtype, nq, nk, heads, hd, ws=False):
    w = heads * hd
    return lib.acid_attention_forward(dtype, p[0], w, p[1], w, p[2], w, p[3], w, nq, nk, heads, hd,
                                      p[4] if ws else None, 1 << 28 if ws else 0, None)
def layernorm(tin, tout, rows, d): return lib.acid_layernorm_mod(tin, p[0], tout, p[1], rows, d, p[2], p[3], 1e-6, None)
def temni(rows, d): return lib.acid_temni_drift(p[0], p[1], p[2], p[3], rows, d, 1e-6, p[4], None, p[5], 1 << 20, None)
EPIS = (A.ACID_EPI_BIAS, A.ACID_EPI_GELU, A.ACID_EPI_GATED_RES, A.ACID_EPI_RES)
"""


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    """The library with the stand-in runtime, and the stand-in itself."""
    from paper_2607_12358_gb300 import build as b

    b.build()
    d = tmp_path_factory.mktemp("runtime")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b.nvcc()))), "include")
    objs = [os.path.join(b.BUILD, s.replace(".cu", ".o")) for s in b.SOURCES]
    src, fake, lib = d / "runtime.cpp", str(d / "libfake.so"), str(d / "libacid.so")

    def cxx(*args):
        subprocess.run(["g++", "-shared", "-fPIC", "-I", cuda, *args], check=True)

    src.write_text(RUNTIME)
    cxx("-o", fake, str(src))
    have = subprocess.run(["nm", "-D", "--defined-only", fake], capture_output=True, text=True, check=True).stdout
    cxx("-o", lib, *objs)
    need = subprocess.run(["nm", "-D", "-u", lib], capture_output=True, text=True, check=True).stdout
    names = {w for w in need.split() if w.startswith(("cuda", "__cuda"))} - {l.split()[-1] for l in have.splitlines()}
    stubs = d / "stubs.c"
    stubs.write_text("".join(f"long {n}() {{ return 0; }}\n" for n in sorted(names)))
    subprocess.run(["gcc", "-c", "-fPIC", "-w", "-o", str(d / "stubs.o"), str(stubs)], check=True)
    cxx("-o", fake, str(src), str(d / "stubs.o"))
    cxx("-o", lib, *objs, fake)
    return lib, fake


def run(script, lib, fake=None, env=None):
    args = [sys.executable, "-c", PRELUDE + script, lib, os.path.join(PKG, "_capi.py")] + ([fake] if fake else [])
    r = subprocess.run(args, capture_output=True, text=True, timeout=300, env=dict(os.environ, **(env or {})))
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])


def test_linear_without_a_usable_device_is_an_error():
    """The whole library on a machine without a GPU: an error code, not the end of the process."""
    from paper_2607_12358_gb300 import build as b

    run("""
for epi in EPIS:
    assert linear(epi=epi) == A.ACID_ERR_CUDA, epi
""", b.build(), env={"CUDA_VISIBLE_DEVICES": ""})


def test_linear_without_a_resident_pair(libs):
    """No pair of CTAs fits, or the query fails: an error each time, and a later query that answers is used."""
    run("""
for epi in EPIS:
    fk.pairs, fk.occupancy_error = 0, 0
    assert linear(epi=epi) == A.ACID_ERR_CUDA
    fk.pairs, fk.occupancy_error = 76, 700
    assert linear(epi=epi) == A.ACID_ERR_CUDA and fk.launches == 0
    fk.occupancy_error = 0
    assert linear(M=32760, epi=epi) == A.ACID_OK
    assert (fk.launches, fk.grid) == (1, 2 * 76)
    fk.launches = 0
""", *libs)


def test_shared_memory_opt_in_on_every_device(libs):
    """Every kernel's opt-in is made on each device that it is launched on, and made again after it failed."""
    run("""
B, F = A.ACID_BF16, A.ACID_FP32
calls = [lambda d=d, i=i, o=o: layernorm(i, o, 5000, d) for d in (520, 1536, 1912, 1920, 3064, 3072) for i in (B, F) for o in (B, F)]
calls += [lambda d=d: temni(5000, d) for d in (512, 1536, 1920, 3072)]
calls += [lambda e=e, o=o: linear(epi=e, out_fp32=o) for e in EPIS for o in (0, 1)]
calls += [lambda m=m: linear(F, M=m, K=256, N=256) for m in (16, 1000, 5000)]
calls += [lambda n=n, h=h: attention(F, n, n, 4, h) for n in (64, 4000) for h in (32, 64, 96, 128)]
calls += [lambda n=n, k=k, h=h: attention(B, n, k, 12, h, True) for n, k in ((4800, 300), (4800, 4800)) for h in (64, 128)]
fk.attribute_error = 1
for i, f in enumerate(calls):
    assert f() in (A.ACID_OK, A.ACID_ERR_CUDA), i  # below 48 KB nothing has to be asked for
fk.attribute_error = 0
for dev in (0, 1, 0):
    fk.device = dev
    for i, f in enumerate(calls):
        assert f() == A.ACID_OK, (dev, i, lib.acid_last_error())
""", *libs)


def test_grids_follow_the_device(libs):
    """Persistent grids are sized to the SMs of the device that the call runs on."""
    run("""
for dev, sms in ((0, 152), (1, 100), (0, 152)):
    fk.device = dev
    assert layernorm(A.ACID_BF16, A.ACID_BF16, 100000, 3072) == A.ACID_OK and fk.grid == 4 * sms
    assert attention(A.ACID_BF16, 30000, 512, 12, 128) == A.ACID_OK and fk.grid == sms
""", *libs)


def test_drift_results_on_another_device_are_copied(libs):
    """The final kernel stores to the caller's outputs where they are memory of the device that it runs on; memory of
    another device, and managed memory, take the copies, which need no peer access."""
    run("""
rel, sums, n = 0x20000000, 0x20000100, 4096 * 3072
calls = [lambda r, s: lib.acid_drift_signal(p[0], p[1], n, A.ACID_BF16, r, s, p[5], 1 << 20, None),
         lambda r, s: lib.acid_drift_apply(p[0], p[1], p[2], p[3], n, A.ACID_BF16, r, s, p[5], 1 << 20, None),
         lambda r, s: lib.acid_temni_drift(p[0], p[1], p[2], p[3], 4096, 3072, 1e-6, r, s, p[5], 1 << 20, None)]
for f in calls:
    for dev, home, kind, stores in ((0, 0, 2, 2), (0, 1, 2, 0), (1, 0, 2, 0), (1, 1, 2, 2), (0, 0, 3, 0)):
        fk.device, fk.home, fk.type, fk.copies, fk.stores = dev, home, kind, 0, 0
        assert f(rel, sums) == A.ACID_OK
        assert (fk.stores, fk.copies) == (stores, 2 - stores), (dev, home, kind, fk.stores, fk.copies)
    fk.device, fk.home, fk.type, fk.copies, fk.stores = 0, 0, 2, 0, 0
    assert f(rel + 4, None) == A.ACID_OK and (fk.stores, fk.copies) == (0, 1)  # not aligned for a double
""", *libs)


def test_scratch_address_after_a_device_reset(libs):
    """The file-scope scratch array is looked up once in each device's context, and again after a reset."""
    run("""
def noalloc(): return lib.acid_drift_signal_noalloc(p[0], p[1], 4096, A.ACID_BF16, 0x20000000, None, None)
for dev, resets, lookups in ((0, 0, 1), (0, 0, 1), (1, 0, 2), (0, 0, 2), (0, 1, 3), (0, 1, 3), (1, 1, 4), (1, 2, 5)):
    fk.device = fk.home = dev
    fk.resets = resets
    assert noalloc() == A.ACID_OK
    assert fk.lookups == lookups, (dev, resets, fk.lookups)
""", *libs)


def test_vectors_that_wide_loads_cannot_read_are_refused(libs):
    """The LayerNorm's vectors and the modulation's weights are read 16 bytes at a time: an address that does not allow
    it is an error before anything is launched."""
    run("""
f = lambda sh, sc: lib.acid_layernorm_mod(A.ACID_FP32, p[0], A.ACID_FP32, p[1], 100, 256, sh, sc, 1e-6, None)
for sh, sc in ((p[2] + 4, p[3]), (p[2], p[3] + 8)):
    assert f(sh, sc) == A.ACID_ERR_UNSUPPORTED and fk.launches == 0
assert f(p[2], p[3]) == A.ACID_OK and f(None, None) == A.ACID_OK and fk.launches == 2
desc = A.acid_block_desc(A.ACID_BLOCK_WAN, A.ACID_FP32, 256, 4, 512, 1, 8, 8, 0, 10000.0, 1e-6)
n = C.c_size_t()
assert lib.acid_block_workspace_size(C.byref(desc), C.byref(n)) == A.ACID_OK
w = A.acid_block_weights()
for name in ("mod", "qkv", "o", "ff1", "ff2"):
    setattr(w, name, A.acid_linear(p[5], p[6]))
cond = A.acid_cond()
cond.temb = p[7]
block = lambda: lib.acid_dit_block_forward(C.byref(desc), p[8], C.byref(cond), C.byref(w), p[9], n.value, None)
assert block() == A.ACID_OK
w.mod = A.acid_linear(p[5] + 8, p[6])
assert block() == A.ACID_ERR_UNSUPPORTED
""", *libs)
