"""Order of the allocation-free entry's kernels behind the one that writes their descriptors.

Host: the entry's object file is linked with launchers that record what they are asked for (no
CUDA runtime), so the flags of every launch are seen without a GPU.  GPU: frames without a detect
region (w or h <= 38) at aligned pitches, as the first calls of a process and after other frames.
"""

import os
import subprocess
import sys

import numpy as np
import pytest

import paper_2506_07164_gb300 as ofg

b = sys.modules[ofg.build.__module__]  # the build module (the package exports its function under the same name)

FAKE = r"""
#include <cstdio>
#include <cstdlib>
#include <string>
#include <cuda_runtime.h>
#include "of_internal.h"
#include "ofast.h"

// What the CUDA compiler's registration and launch code calls.
static char device_array[1 << 10];
extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void*) { *k = nullptr; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { std::puts("setup 0"); return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return ""; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = device_array; return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
    std::puts("copy 0");
    return cudaSuccess;
}
}
namespace ofk {
void set_last_error(const std::string&) {}
void set_select_smem_limit(int) {}
int select_smem_bytes(int) { return 0; }
int encode_u8_map(CUtensorMap*, const void*, int, int, int, int, int) { return OF_OK; }
int fast_blocks_per_sm() { return 1; }
int nms_blocks_per_sm() { return 1; }
void launch_fast(const Img*, const int32_t*, const int32_t*, int, int n_tiles, const CUtensorMap*, const Call*, int, int,
                 int, int, int, int, void*, bool, int) {
    if (n_tiles > 0) std::puts("fast 0");
}
void launch_nms_harris(const Img*, const int32_t*, const int32_t*, int, int n_tiles, const CUtensorMap*,
                       const CUtensorMap*, const Call*, int, int, int, int, int, int, void*, bool, int, bool pdl) {
    if (n_tiles > 0) std::printf("nms %d\n", pdl);
}
void launch_select(const Img*, int, int, const Call*, int, bool, void*, bool pdl) { std::printf("select %d\n", pdl); }
void launch_orient(const Img*, int, const Call*, int total_slots, bool, bool, void*, bool pdl) {
    if (total_slots > 0) std::printf("orient %d\n", pdl);
}
}  // namespace ofk
int main(int, char** a) {
    const int w = std::atoi(a[1]), h = std::atoi(a[2]), pitch = std::atoi(a[3]), n = std::atoi(a[4]);
    return of_detect_level_noalloc((const uint8_t*)4096, w, h, pitch, 20, 7, 0.04f, n, (of_keypoint*)8192, (int32_t*)12288,
                                   nullptr);
}
"""


@pytest.fixture(scope="module")
def recorder(tmp_path_factory):
    b.build()
    d = tmp_path_factory.mktemp("fake")
    (d / "fake.cpp").write_text(FAKE)
    exe = str(d / "fake")
    cuda = os.path.dirname(os.path.dirname(b._nvcc()))
    r = subprocess.run(["g++", "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", b.INCLUDE, "-I", b.CSRC,
                        str(d / "fake.cpp"), os.path.join(b.BUILD, "of_noalloc.cu.o"),
                        os.path.join(b.BUILD, "of_plan.cpp.o"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("w,h,pitch,n", [(640, 480, 640, 500), (641, 480, 641, 500), (32, 32, 32, 300), (38, 200, 48, 300),
                                         (200, 38, 208, 300), (30, 30, 30, 300), (32, 32, 32, 0), (640, 480, 640, 0)])
def test_first_kernel_waits_for_the_descriptors(recorder, w, h, pitch, n):
    """Only a kernel whose predecessor on the stream is another kernel of the chain may start early: the
    first one behind the setup kernel (or the copy) reads descriptors before its own wait."""
    r = subprocess.run([recorder, *map(str, (w, h, pitch, n))], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    steps = [tuple(s.split()) for s in r.stdout.splitlines()]
    names = [s[0] for s in steps]
    empty = w <= 38 or h <= 38
    assert names == ["setup"] + ["copy"] * (pitch % 16 != 0) + ["fast", "nms"] * (not empty) + ["select"] + \
        ["orient"] * (n > 0)
    first = 1 + (pitch % 16 != 0)
    assert steps[first][1] == "0", steps


EMPTY = r"""
import sys
import torch
import paper_2506_07164_gb300 as ofg
n = 300
out = torch.full((n * 64,), 77, dtype=torch.uint8, device="cuda")
cnt = torch.full((1,), -1, dtype=torch.int32, device="cuda")
for w, h, pitch in ((32, 32, 32), (208, 32, 208), (38, 200, 48)):
    t = torch.zeros((h, pitch), dtype=torch.uint8, device="cuda")
    cnt.fill_(-1)
    ofg.of_detect_level_noalloc(t, w, h, pitch, 20, 7, 0.04, n, out, cnt)
    torch.cuda.synchronize()
    assert int(cnt) == 0, (w, h, int(cnt))
assert bool((out == 77).all())
print("empty ok")
"""


@pytest.mark.gpu
def test_first_call_of_a_process_without_a_detect_region():
    r = subprocess.run([sys.executable, "-c", EMPTY], capture_output=True, text=True, cwd=b.ROOT, timeout=300)
    assert r.returncode == 0 and "empty ok" in r.stdout, r.stdout + r.stderr


@pytest.mark.gpu
def test_no_detect_region_after_a_frame_with_one():
    torch = pytest.importorskip("torch")
    import synth

    n = 300
    big = torch.from_numpy(synth.scene(640, 480, 31)).cuda()
    out = torch.zeros(n * 64, dtype=torch.uint8, device="cuda")
    other = torch.full((n * 64,), 77, dtype=torch.uint8, device="cuda")
    cnt = torch.zeros(2, dtype=torch.int32, device="cuda")
    tiny = torch.from_numpy(np.ascontiguousarray(synth.scene(208, 32, 32))).cuda()
    for _ in range(5):  # back to back: the empty frame's kernels see their own outputs and counters
        ofg.of_detect_level_noalloc(big, 640, 480, 640, 20, 7, 0.04, n, out, cnt[:1])
        ofg.of_detect_level_noalloc(tiny, 208, 32, 208, 20, 7, 0.04, n, other, cnt[1:])
    torch.cuda.synchronize()
    assert cnt.tolist() == [n, 0]
    assert bool((other == 77).all())
