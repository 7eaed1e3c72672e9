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

extern "C" {
// what the stand-in answers
int fk_pairs = 76, fk_occupancy_error = 0;
// what it was asked
int fk_launches = 0, fk_grid = 0;

cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = fk_pairs;
  return (cudaError_t)fk_occupancy_error;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**) {
  ++fk_launches;
  fk_grid = (int)c->gridDim.x;
  return cudaSuccess;
}
static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                       const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** fn, unsigned int, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *fn = !std::strcmp(name, "cuTensorMapEncodeTiled") ? (void*)encode : nullptr;
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
