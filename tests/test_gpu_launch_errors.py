"""A launch that the runtime refuses ends the call with an error, and by then the
work that the call had already enqueued is done: the caller's buffers are idle.
(A configuration of 4096 threads per block is refused on the host.)"""
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#include "he_internal.h"
// sets the flag about 20 ms after its start
__global__ void k_late(volatile int *flag) {
    const long long t0 = clock64();
    for (int i = 0; i < 1 << 24 && clock64() - t0 < 40000000ll; i++) {}
    *flag = 1;
    __threadfence_system();
}
__global__ void k_next() {
    pdl_trigger();
    pdl_wait();
}
int main() {
    int *h = nullptr, *d = nullptr;
    cudaStream_t st;
    if (cudaHostAlloc((void **)&h, sizeof(int), cudaHostAllocMapped) != cudaSuccess) return 2;
    if (cudaHostGetDevicePointer((void **)&d, h, 0) != cudaSuccess) return 2;
    if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) return 2;
    he::launch_pdl(k_next, dim3(1), 32, 0, st);   // loads the module
    cudaStreamSynchronize(st);
    *h = 0;
    k_late<<<1, 1, 0, st>>>(d);
    int at_error = -1;
    try {
        he::launch_pdl(k_next, dim3(1), 4096, 0, st);
    } catch (const he::HeError &e) {
        at_error = *(volatile int *)h;
    }
    cudaStreamSynchronize(st);
    printf("at_error %d after %d\n", at_error, *(volatile int *)h);
    return 0;
}
"""


def test_a_refused_launch_leaves_nothing_running(tmp_path):
    from paper_2305_17341_gb300 import builder
    src, exe = tmp_path / "launch.cu", tmp_path / "launch"
    src.write_text(SOURCE)
    subprocess.run([builder.nvcc()] + builder.ARCH + ["-O1", "-std=c++17", "-I", builder.CSRC, "-I", builder.INCLUDE,
                                                      "-o", str(exe), str(src)], check=True, timeout=300)
    out = subprocess.run([str(exe)], check=True, timeout=60, capture_output=True, text=True).stdout
    assert out.split() == ["at_error", "1", "after", "1"], out
