"""A kernel that the driver refuses to launch does not fail a call that another kernel covers.  The library's objects are linked
against a stand-in for the CUDA runtime that refuses the launches of one kernel and names the others; nothing runs on a GPU."""
import os
import subprocess

import pytest

from paper_2110_14871_b200 import build as gbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OBJECTS = os.path.join(ROOT, "paper_2110_14871_b200", "_build")

PROGRAM = r"""
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <map>
#include <string>
#include "gdws.h"

static std::map<const void *, std::string> &names() { static std::map<const void *, std::string> m; return m; }
static const char *refused = "";
static int registers = 80;
static std::string launched;

static cudaError_t launch(const void *f)
{
    const std::string &n = names()[f];
    if (*refused && n.find(refused) != std::string::npos) return cudaErrorLaunchOutOfResources;
    launched += n + " ";
    return cudaSuccess;
}
static CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *f, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) { names()[f] = name; }
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t, cudaStream_t) { return launch(f); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *f, void **) { return launch(f); }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int) { *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : 148; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *, const void *, size_t, enum cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, enum cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "refused"; }
cudaError_t cudaFuncSetAttribute(const void *, enum cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *) { memset(a, 0, sizeof(*a)); a->numRegs = registers; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c) { *n = 120 / (int)c->attrs[0].val.clusterDim.x; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char *, void **f, unsigned long long, enum cudaDriverEntryPointQueryResult *r) { *f = (void *)encode; *r = cudaDriverEntryPointSuccess; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) { static char z[256]; *p = z; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes *a, const void *) { memset(a, 0, sizeof(*a)); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *, cudaEvent_t, cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
}

// call, refused kernel, registers that every kernel is said to have
int main(int, char **argv)
{
    const std::string call = argv[1];
    refused = argv[2];
    registers = atoi(argv[3]);
    const int C = 256, D = 256, H = 14, N = call == "f32" || call == "stage" ? 16 : 1;
    int32_t g[C];
    for (int &v : g) v = 3;
    gdws_plan_t *plan = nullptr;
    if (gdws_plan(C, D, 3, 1, 1, g, &plan) != GDWS_OK) return 2;
    char *mem = (char *)(uintptr_t)0x10000000;          // never read
    const bool f32 = call == "f32";
    gdws_tensor_t x = {mem, f32 ? GDWS_F32 : GDWS_BF16, GDWS_NHWC, N, C, H, H}, y = x;
    y.ptr = mem + (64 << 20);
    y.c = D;
    void *w = mem + (128 << 20);
    if (!f32 && gdws_pack_weights(plan, w, w, nullptr, GDWS_BF16, nullptr) != GDWS_OK) return 3;
    launched.clear();
    const gdws_status_t st = call == "stage" ? gdws_depthwise(plan, &x, nullptr, y.ptr, nullptr) : gdws_forward(plan, &x, f32 ? w : nullptr, f32 ? w : nullptr, nullptr, &y, nullptr);
    printf("%d %s\n", (int)st, launched.c_str());
    gdws_destroy(plan);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gbuild.build_library()
    if not os.path.exists(os.path.join(OBJECTS, "api.o")):
        gbuild.build_library(force=True)
    d = tmp_path_factory.mktemp("refused")
    (d / "p.cpp").write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(gbuild._nvcc())), "include")
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", cuda, str(d / "p.cpp"),
                           *(os.path.join(OBJECTS, s.replace(".cu", ".o")) for s in gbuild.SOURCES), "-o", str(d / "p"), "-lpthread"])
    return str(d / "p")


@pytest.mark.parametrize("call,refused,registers,kernel", [
    ("f32", "", 80, "f32_tc_kernel"), ("f32", "f32_tc_kernel", 80, "fused_f32_kernel"), ("f32", "", 72, "fused_f32_kernel"),
    ("stage", "", 80, "gdw_tc_kernel"), ("stage", "gdw_tc_kernel", 80, "fused_bf16_kernel"),
    ("folded", "", 80, "fold_split_kernel"), ("folded", "fold_split_kernel", 80, "fold_kernel"),
])
def test_another_kernel_takes_the_call(program, call, refused, registers, kernel):
    out = subprocess.run([program, call, refused, str(registers)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out
    status, *launched = out.stdout.split()
    assert status == "0" and len(launched) == 1 and kernel in launched[0], out.stdout


def test_no_kernel_is_a_status(program):
    out = subprocess.run([program, "f32", "f32", "80"], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.split() == ["4"], out
