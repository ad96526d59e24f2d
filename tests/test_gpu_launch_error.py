"""A launch that the CUDA runtime refuses is reported by the launcher and by nothing
after it: no stale error is left for the next caller of cudaGetLastError.  launch_pdl is
taken from mfc_launch.cuh; the refused launch asks for more threads than a block may
have, which the runtime answers without reaching the GPU."""
import os
import re
import subprocess

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
LAUNCH = os.path.join(HERE, os.pardir, "paper_2305_09163_gb300", "csrc", "mfc_launch.cuh")
MAIN = """
#include <cstdio>
#include <cuda_runtime.h>
%s
__global__ void one(int* p) { *p = 1; }
int main() {
    int *p = nullptr, h = 0;
    if (cudaMalloc(&p, sizeof *p) != cudaSuccess) return 1;
    cudaMemset(p, 0, sizeof *p);
    const cudaError_t refused = launch_pdl(one, 1u, 4096, 0, nullptr, p), stale = cudaGetLastError();
    const cudaError_t taken = launch_pdl(one, 1u, 1, 0, nullptr, p);
    cudaMemcpy(&h, p, sizeof h, cudaMemcpyDeviceToHost);
    std::printf("%%d %%d %%d %%d\\n", (int)refused, (int)stale, (int)taken, h);
    return 0;
}
"""


def test_refused_launch_is_reported_once(tmp_path):
    with open(LAUNCH) as f:
        fn = re.search(r"template <[^>]*>\ncudaError_t launch_pdl\(.*?\n}\n", f.read(), re.S).group(0)
    src, exe = str(tmp_path / "t.cu"), str(tmp_path / "t")
    with open(src, "w") as f:
        f.write(MAIN % fn)
    from paper_2305_09163_gb300 import _build
    subprocess.run([_build._nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", src, "-o", exe], check=True)
    refused, stale, taken, value = map(int, subprocess.run([exe], check=True, capture_output=True, text=True,
                                                            timeout=60).stdout.split())
    assert refused != 0 and stale == 0 and taken == 0 and value == 1
