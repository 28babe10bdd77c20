"""Bounded mbarrier waits of the tensor-core kernels: a wait whose result a
whole warp acts on (tcgen05.ld, shuffles) gives one result to all its lanes."""
import ctypes
import glob
import os
import re
import subprocess

import numpy as np
import pytest

from paper_2211_14318_gb300 import build as b


def _guards(src: str):
    """(line, headers of the enclosing blocks) of each plain mbar_wait call."""
    src = re.sub(r"/\*.*?\*/", " ", re.sub(r"//[^\n]*", "", src), flags=re.S)
    stack, start = [], 0
    for m in re.finditer(r"[{};]|\bmbar_wait\(", src):
        t = m.group()
        if t == "{":
            stack.append(src[start:m.start()])
        elif t == "}":
            stack.pop()
        if t in "{};":
            start = m.end()
        else:
            yield src.count("\n", 0, m.start()) + 1, list(stack)


def test_warps_take_one_branch_after_a_wait():
    found = 0
    for path in sorted(glob.glob(os.path.join(b.CSRC, "*.cu"))):
        for line, blocks in _guards(open(path).read()):
            found += 1
            assert any("lane == 0" in h or "threadIdx.x == 0" in h for h in blocks), \
                f"{os.path.basename(path)}:{line}: a per-lane wait outside a single lane's code"
    assert found > 10  # the issuing lanes' own waits


SRC = r"""
#include "cvx_tc.cuh"
using namespace cvx;
// Warp 0 waits with a limit of lane x step ns (or limit, if longer), warp 1
// arrives after delay ns: ok[lane] the warp's result, ok[32 + lane] that of a
// second barrier's plain wait.
__global__ void k(unsigned long long step, unsigned long long limit, unsigned long long delay, int *ok) {
    __shared__ __align__(8) uint64_t bar[2];
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    for (int i = 0; i < 2; ++i) {
        if (threadIdx.x < 32) {
            const unsigned long long l = lane * step > limit ? lane * step : limit;
            const bool r = i == 0 ? mbar_wait_warp(&bar[0], 0, l) : mbar_wait(&bar[1], 0, l);
            ok[32 * i + lane] = r ? 1 : 0;
        } else if (lane == 0) {
            const uint64_t t0 = global_ns();
            while (global_ns() - t0 < delay) {
            }
            mbar_arrive(&bar[i]);
        }
        __syncthreads();
    }
}
extern "C" int run(unsigned long long step, unsigned long long limit, unsigned long long delay, int *ok) {
    int *d = nullptr;
    cudaError_t e = cudaMalloc(&d, 64 * sizeof(int));
    if (e != cudaSuccess) return (int)e;
    k<<<1, 64>>>(step, limit, delay, d);
    e = cudaMemcpy(ok, d, 64 * sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
"""


@pytest.mark.gpu
def test_wait_result_is_one_per_warp(tmp_path):
    src, so = tmp_path / "w.cu", tmp_path / "w.so"
    src.write_text(SRC)
    subprocess.run([b.nvcc(), "-O2", "-std=c++17", *b.ARCH, "-Xcompiler", "-fPIC", "-I", b.CSRC,
                    "-shared", "-cudart", "static", "-o", str(so), str(src)], check=True)
    run = ctypes.CDLL(str(so)).run
    run.argtypes = [ctypes.c_uint64] * 3 + [ctypes.c_void_p]
    ok = np.full(64, -1, np.int32)
    # limits 0 .. 62 ms, arrival after 30 ms: a lane's own wait may go either way
    assert run(2000000, 0, 30000000, ok.ctypes.data) == 0
    assert ok[:32].tolist() in ([0] * 32, [1] * 32)
    # nothing arrives before the limit; arrival long before it
    assert run(0, 2000000, 60000000, ok.ctypes.data) == 0
    assert ok.tolist() == [0] * 64
    assert run(0, 1000000000, 400000, ok.ctypes.data) == 0
    assert ok.tolist() == [1] * 64
