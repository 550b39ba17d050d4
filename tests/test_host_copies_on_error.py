"""pic_render_host when a CUDA call fails half-way: the library's host code, compiled against a stand-in for the CUDA runtime that
counts what is in flight on each stream and fails the call it is told to.  No copy into the caller's memory may be under way
on a stream that the caller cannot wait for when the call returns."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_26005_b200", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

FAKE = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include "pic_types.h"
#include "../../include/pictura.h"

static int g_calls = 0, g_fail_at = -1, g_in_flight = 0, g_chunks = 0;       // counted: what pic_render_host asks of the private stream
static cudaStream_t g_private = nullptr;
static cudaError_t tick() { return g_calls++ == g_fail_at ? cudaErrorUnknown : cudaSuccess; }

extern "C" {
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) { std::memset(p, 0, sizeof(*p)); p->major = 10; p->sharedMemPerBlockOptin = 232448; p->multiProcessorCount = 148; return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::malloc(n); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind kind, cudaStream_t s) {
    if (kind != cudaMemcpyDeviceToHost || s != g_private) return cudaSuccess;
    const cudaError_t e = tick();
    if (e == cudaSuccess) ++g_in_flight;
    return e;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = g_private = reinterpret_cast<cudaStream_t>(0x1000); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { if (s == g_private) g_in_flight = 0; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { ++g_chunks; return tick(); }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(0x2000); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }
}

namespace pic {
size_t max_smem_bytes() { return 0; }
cudaError_t configure_kernels() { return cudaSuccess; }
cudaError_t launch_setup(const RenderParams&, int, const float*, float*, const float*, const float*, const uint8_t*, const uint8_t*, AgentGeom*, ViewCam*, uint32_t*,
                         float, float, float, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_render(const RenderParams&, long long, bool, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_colour(const RenderParams&, long long, bool, int, cudaStream_t) { return cudaSuccess; }
size_t survivor_bytes_per_tile() { return 2048; }
}

int main() {
    pic_scene_desc d = {};
    const int64_t offset[2] = {0, 0};
    d.size = sizeof(d); d.E = 1; d.A = 8; d.K = 1; d.H = 1024; d.W = 1024; d.near_z = 0.5f; d.far_z = 100.f; d.num_maps = 1; d.map_tri_offset = offset;
    pic_scene* s = nullptr;
    if (pic_scene_create(&d, &s) != PIC_OK) return std::printf("create: %s\n", pic_last_error()), 1;
    const size_t px = 8u << 20;
    std::vector<float> poses(24, 0.f), dims(24, 1.f);
    std::vector<uint8_t> cls(px);
    std::vector<uint16_t> dep(px);
    const pic_camera cam = {0.f, 0.f, 1.f, 0.f, 0.f, 100.f, 100.f};
    int total = 0;
    for (int fail_at = -1; fail_at < (total ? total : 1); ++fail_at) {
        g_calls = 0; g_in_flight = 0; g_chunks = 0; g_fail_at = fail_at;
        const pic_status st = pic_render_host(s, poses.data(), dims.data(), nullptr, &cam, cls.data(), dep.data(), reinterpret_cast<void*>(0x3000));
        if (fail_at < 0) {
            total = g_calls;
            if (st != PIC_OK || g_chunks < 2 || total < 6) return std::printf("%d parts, %d calls, status %d\n", g_chunks, total, st), 1;
        } else if (st != PIC_ERR_CUDA) {
            return std::printf("call %d failed, status %d\n", fail_at, st), 1;
        }
        if (g_in_flight) return std::printf("call %d failed: %d copies still under way at the return\n", fail_at, g_in_flight), 1;
    }
    pic_scene_destroy(s);
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")), reason="needs g++ and the CUDA headers")
def test_no_copy_outlives_a_failed_call(tmp_path):
    src, exe = tmp_path / "fake.cpp", tmp_path / "fake"
    src.write_text(FAKE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CUDA, "-I", CSRC, "-x", "c++", str(src), os.path.join(CSRC, "pic_api.cu"),
                    os.path.join(CSRC, "pic_bvh.cpp"), "-pthread", "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
