"""Which copy ld_pack_planes / ld_unpack_planes make, without a GPU: ld_api.cu
compiled against a fake CUDA runtime that says where pointers and streams
live. The copy kernel only where buffer, state, stream and current device are
one GPU's; the runtime's copy, which any device's stream takes, everywhere
else."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1609_01479_gb300", "csrc")

FAKE = r"""
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include "ld.h"
#include "ld_internal.h"

static int g_current, g_kernel, g_runtime;
struct Range { uintptr_t lo, hi; cudaPointerAttributes a; };
static Range g_ranges[2];  // the workspace and the buffer

extern "C" {
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    for (const Range& r : g_ranges)
        if ((uintptr_t)p >= r.lo && (uintptr_t)p < r.hi) return *a = r.a, cudaSuccess;
    return cudaErrorInvalidValue;
}
cudaError_t cudaGetDevice(int* d) { return *d = g_current, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
    return ++g_runtime, cudaSuccess;
}
}
namespace ld {
cudaError_t launch_copy_rows(void*, size_t, const void*, size_t, size_t, int, cudaStream_t s) {
    if (s && (int)(uintptr_t)s - 1 != g_current) return cudaErrorInvalidResourceHandle;  // the NULL stream: the current device's
    return ++g_kernel, cudaSuccess;
}
cudaError_t launch_default_refs(ld_ctx*) { return cudaSuccess; }
int choose_step_kernel(int, int, int, int, int, int) { return kStepGeneric; }
namespace lp {
cudaError_t init(ld_ctx*, const double*, const double*, const double*, const double*) { return cudaSuccess; }
}
}  // namespace ld

// argv: device of the state, of the buffer, current device, stream (0: NULL, else device + 1), buffer managed.
// Prints kernel and runtime copies of one pack and one unpack.
int main(int, char** v) {
    ld_params p{};
    p.tau_f = p.tau_g = 1.0, p.rho0 = 1.0, p.precision = LD_FP32;
    p.stencil = LD_STENCIL_7, p.force = LD_FORCE_POTENTIAL, p.collision = LD_COLLISION_BGK, p.rounding = LD_ROUND_NEAREST;
    const size_t bytes = ld_workspace_bytes(4, 4, 4, &p);
    char* ws = (char*)aligned_alloc(256, bytes);
    char* buf = (char*)aligned_alloc(256, 1 << 16);
    g_ranges[0] = {(uintptr_t)ws, (uintptr_t)ws + bytes, {cudaMemoryTypeDevice, atoi(v[1]), ws, nullptr}};
    g_ranges[1] = {(uintptr_t)buf, (uintptr_t)buf + (1 << 16),
                   {atoi(v[5]) ? cudaMemoryTypeManaged : cudaMemoryTypeDevice, atoi(v[2]), buf, nullptr}};
    g_current = atoi(v[3]);
    ld_ctx* c = nullptr;
    if (ld_create(4, 4, 4, &p, ws, bytes, (void*)(uintptr_t)atoi(v[4]), &c)) return puts(ld_last_error(nullptr)), 1;
    if (ld_init(c, (const double*)buf, nullptr, nullptr)) return puts(ld_last_error(c)), 1;
    if (ld_pack_planes(c, 1, 2, buf) || ld_unpack_planes(c, 1, 2, buf)) return puts(ld_last_error(c)), 1;
    printf("%d %d\n", g_kernel, g_runtime);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no CUDA headers")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    out = tmp_path_factory.mktemp("planes")
    (out / "fake.cpp").write_text(FAKE)
    exe = str(out / "planes")
    # what the calls of this program do not reach is left unresolved
    subprocess.run(["g++", "-std=c++17", "-I", inc, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-x", "c++",
                    os.path.join(CSRC, "ld_api.cu"), str(out / "fake.cpp"), "-o", exe, "-ldl",
                    "-Wl,--unresolved-symbols=ignore-all"], check=True, capture_output=True, text=True)
    return exe


@pytest.mark.parametrize("state,buf,current,stream,managed,kernel", [
    (0, 0, 0, 0, 0, True),    # the ordinary call: NULL stream
    (0, 0, 0, 1, 0, True),    # a stream of GPU 0
    (1, 1, 1, 2, 0, True),
    (1, 1, 0, 0, 0, False),   # GPU 1's lattice while GPU 0 is current, NULL stream
    (1, 1, 0, 2, 0, False),   # the same on a stream of GPU 1
    (0, 0, 0, 2, 0, False),   # a stream of another GPU
    (0, 1, 0, 1, 0, False),   # the buffer on another GPU
    (1, 0, 0, 1, 0, False),
    (0, 0, 0, 1, 1, False),   # managed memory
])
def test_copy_route(program, state, buf, current, stream, managed, kernel):
    args = [str(a) for a in (state, buf, current, stream, managed)]
    out = subprocess.run([program, *args], check=True, capture_output=True, text=True).stdout
    assert out.split() == (["2", "0"] if kernel else ["0", "2"])
