"""A step launch that the runtime refuses (here a block of 4096 threads: an invalid
configuration, found on the host) is reported to its own caller and to no later
launch: the runtime's last error is clear afterwards and a valid launch succeeds."""
import subprocess

import pytest

from paper_1912_00695_gb300 import build

pytestmark = pytest.mark.gpu

SRC = """#include <cstdio>
#include "fd_launch_count.h"
#include "fd_tma.cuh"
using namespace fdgb;
namespace fdgb {
int count = 0;
void count_launches(cudaStream_t, int n) { count += n; }
}
__global__ void kernel(int *out) { if (threadIdx.x == 0) *out = 7; }
int main() {
    int *out = nullptr, got = 0;
    if (cudaMalloc(&out, 4) != cudaSuccess) return 1;
    int bad = 0;
    for (bool overlap : {false, true}) {
        const cudaError_t refused = counted(launch_step(kernel, dim3(1), 4096, 0, overlap, nullptr, out), nullptr);
        const cudaError_t left = cudaPeekAtLastError();
        const cudaError_t next = counted(launch_step(kernel, dim3(1), 32, 0, overlap, nullptr, out), nullptr);
        std::printf("refused %d left %d next %d\\n", int(refused), int(left), int(next));
        bad |= refused == cudaSuccess || left != cudaSuccess || next != cudaSuccess;
    }
    if (cudaMemcpy(&got, out, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    return bad || got != 7 || count != 2 ? 3 : 0;
}
"""


def test_a_refused_launch_is_reported_once(tmp_path):
    (tmp_path / "t.cu").write_text(SRC)
    subprocess.run([build.nvcc(), str(tmp_path / "t.cu"), "-o", str(tmp_path / "t")] + build.NVCC_FLAGS, check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
