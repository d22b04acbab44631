"""Giving a pool's block back (rs_block.cuh) on a fake CUDA runtime of two
devices: the wait and the free happen on the block's device, whatever device
the calling thread has current, which it keeps."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1110_4372_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "rs_block.cuh"
static int current;
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { current = d; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { printf("wait %d,", current); return cudaSuccess; }
cudaError_t cudaFree(void *) { printf("free %d,", current); return cudaSuccess; }
}
int main(int, char **argv)
{
    current = atoi(argv[1]);
    rs_block_give_back(argv[3][0] == 'p' ? argv : nullptr, atoi(argv[2]));
    printf("now %d", current);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime_api.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("block")
    src, exe = d / "block.cpp", d / "block"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", f"-I{CSRC}", f"-I{cuda}/include", str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("current,device", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_waits_and_frees_on_the_blocks_device(program, current, device):
    out = subprocess.run([program, str(current), str(device), "p"], check=True, capture_output=True, text=True).stdout
    assert out == f"wait {device},free {device},now {current}"


def test_nothing_to_free(program):
    out = subprocess.run([program, "0", "1", "0"], check=True, capture_output=True, text=True).stdout
    assert out == "now 0"
