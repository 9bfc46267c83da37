"""What the activation quantizer and the row sums ask the CUDA runtime for, seen from the runtime: the library's own sources are linked with
a runtime that launches nothing and writes down every launch (no GPU)."""
import ctypes
import subprocess

import pytest

import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import build as qb_build

FAKE_RUNTIME = r"""
#include <cuda_runtime_api.h>
#include <map>
#include <string>
#include <vector>

struct Launch { std::string name; int l1; };
static std::map<const void*, std::string>& names() {  // filled while the other sources are set up
  static std::map<const void*, std::string> m;
  return m;
}
static std::map<const void*, int> of_function;  // a kernel's own preference, where one was set
static std::vector<Launch> launches;

extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[host] = name;
}
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaErrorUnknown; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : a == cudaDevAttrMultiProcessorCount ? 148 : 0;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPoint(const char*, void**, unsigned long long, cudaDriverEntryPointQueryResult*) { return cudaErrorUnknown; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaErrorUnknown; }
static bool refuse;
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a != cudaFuncAttributePreferredSharedMemoryCarveout) return cudaSuccess;
  if (refuse) return cudaErrorInvalidValue;
  of_function[f] = v;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  int l1 = of_function.count(f) && of_function[f] == cudaSharedmemCarveoutMaxL1;
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributePreferredSharedMemoryCarveout)
      l1 = c->attrs[i].val.sharedMemCarveout == cudaSharedmemCarveoutMaxL1;
  launches.push_back({names()[f], l1});
  return cudaSuccess;
}
int fake_launches() { return (int)launches.size(); }
const char* fake_name(int i) { return launches[i].name.c_str(); }
int fake_l1(int i) { return launches[i].l1; }
void fake_clear() { launches.clear(); }
void fake_refuse(int r) { refuse = r; }
int fake_functions_set() { return (int)of_function.size(); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fake_runtime")
    (d / "runtime.cpp").write_text(FAKE_RUNTIME)
    qb_build.build()
    nvcc = [qb_build._nvcc(), "-std=c++17", "-O3", "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC",
            "-I", str(qb_build.INCLUDE), "-I", str(qb_build.CSRC)]
    objects, procs = [], [subprocess.Popen([*nvcc, "-c", str(d / "runtime.cpp"), "-o", str(d / "runtime.o")])]
    for source in ("api.cu", "quantize_act.cu", "gemm.cu"):
        obj = qb_build.PKG / "_build" / (source + ".o")
        if qb_build._stale(obj, "*.cu", "*.cuh"):  # a library that came without its objects
            obj = d / (source + ".o")
            procs.append(subprocess.Popen([*nvcc, "-c", str(qb_build.CSRC / source), "-o", str(obj)]))
        objects.append(str(obj))
    assert all([p.wait() == 0 for p in procs])
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic,-z,defs", "-o", str(d / "fake.so"), str(d / "runtime.o"), *objects], check=True)
    lib = ctypes.CDLL(str(d / "fake.so"))
    lib.fake_name.restype = ctypes.c_char_p
    return lib


def launches(lib, call):
    """(kernel, whether its launch asks for the SM's cache as L1) of each launch of a call"""
    lib.fake_clear()
    assert call() == qb.QB_OK
    return [(lib.fake_name(i).decode(), bool(lib.fake_l1(i))) for i in range(lib.fake_launches())]


def quantize(lib, M, K):
    p = ctypes.c_void_p
    return lib.qb_quantize_act(p(1 << 32), ctypes.c_int64(M), ctypes.c_int64(K), p(2 << 32), p(3 << 32), p(4 << 32), p(5 << 32),
                               ctypes.c_size_t(1 << 20), p(0))


def quantize_batch(lib, shapes):
    descs = (qb.ActDescC * len(shapes))()
    for d, (M, K) in zip(descs, shapes):
        d.x, d.M, d.K, d.xq, d.act_scale, d.rowsum = 1 << 32, M, K, 2 << 32, 3 << 32, 4 << 32
    return lib.qb_quantize_act_batch(descs, len(shapes), ctypes.c_void_p(5 << 32), ctypes.c_size_t(1 << 20), ctypes.c_void_p(0))


def rowsum(lib, M, K):
    p = ctypes.c_void_p
    return lib.qb_rowsum_i8(p(1 << 32), ctypes.c_int64(M), ctypes.c_int64(K), p(2 << 32), p(0))


def test_a_preference_neither_fails_a_call_nor_outlasts_it(lib):
    calls = (lambda: quantize(lib, 6000, 768), lambda: quantize_batch(lib, [(128, 768)] * 3), lambda: rowsum(lib, 6000, 768))
    for refuse in (1, 0):
        lib.fake_refuse(refuse)
        for call in calls:
            assert all(l1 for _, l1 in launches(lib, call))
            assert lib.fake_functions_set() == 0  # nothing that later launches of the process would find


def test_both_passes_ask_for_l1(lib):
    for _ in range(2):
        for call in (lambda: quantize(lib, 6000, 768), lambda: quantize_batch(lib, [(128, 768), (128, 3072)])):
            got = launches(lib, call)
            assert len(got) == 2 and "act_absmax_kernel" in got[0][0] and "act_quantize_kernel" in got[1][0]
            assert got[0][1] and got[1][1], got


def test_one_launch_asks_for_nothing(lib):
    for M in (32, 1024):
        (name, l1), = launches(lib, lambda: quantize(lib, M, 768))
        assert "act_fused_kernel" in name and not l1
