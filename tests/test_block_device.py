"""A context's memory pool and its blocks (rs_block.cuh) on a fake CUDA runtime
of two devices: the wait and the free of a block happen on the block's device,
whatever device the calling thread has current, which it keeps; and the pool
is destroyed by whoever lets go of it last, the context or a block."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1110_4372_gb300", "csrc")

# argv: the current device, the pool's device, and letters: a (a block is taken), f (one is given back), n (a null
# one is), c (the context goes)
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "rs_block.cuh"
static int current;
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { current = d; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { printf("wait%d ", current); return cudaSuccess; }
cudaError_t cudaFreeAsync(void *, cudaStream_t) { printf("free%d ", current); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { printf("done%d ", current); return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { printf("destroy "); return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t n) { printf("trim%d ", (int)n); return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *v)
{
    printf("keep%d ", (int)*(unsigned long long *)v);
    return cudaSuccess;
}
}
int main(int, char **argv)
{
    current = atoi(argv[1]);
    RsPool *pool = new RsPool();
    pool->device = atoi(argv[2]);
    for (const char *s = argv[3]; *s; s++) {
        if (*s == 'a') pool->holders.fetch_add(1);
        if (*s == 'f') rs_block_give_back(argv, pool);
        if (*s == 'n') rs_block_give_back(nullptr, nullptr);
        if (*s == 'c') rs_pool_retire(pool);
    }
    printf("on%d", current);
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
    return lambda *a: subprocess.run([str(exe), *map(str, a)], check=True, capture_output=True, text=True).stdout


@pytest.mark.parametrize("current,device", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_waits_and_frees_on_the_blocks_device(program, current, device):
    assert program(current, device, "af") == f"wait{device} free{device} done{device} on{current}"


def test_nothing_to_free(program):
    assert program(0, 1, "n") == "on0"


@pytest.mark.parametrize("steps,out", [
    ("c", "keep0 trim0 destroy on0"),
    ("afc", "wait0 free0 done0 keep0 trim0 destroy on0"),
    ("aacff", "keep0 trim0 wait0 free0 done0 wait0 free0 done0 destroy on0"),
    ("aafcf", "wait0 free0 done0 keep0 trim0 wait0 free0 done0 destroy on0")])
def test_the_last_holder_destroys_the_pool(program, steps, out):
    assert program(0, 0, steps) == out
