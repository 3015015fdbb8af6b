"""The first Linear and Q K^T calls of a process, made by many host threads at once: each of them succeeds and
writes the same bytes as a later call (the driver's tensor-map encoder is looked up once, by whichever is first)."""
import os
import subprocess
from pathlib import Path

import pytest
import torch

from paper_2111_13824_gb300 import build as fbuild

pytestmark = pytest.mark.gpu

_PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <cstring>
#include <thread>
#include <vector>
#include <cuda_runtime.h>
#include "fqvit.h"

constexpr int T = 12, M = 96, N = 64, K = 64, L = 144, LD = 144;

struct Call {
    uint8_t *y;
    int8_t *logits;
    void *ws;
    cudaStream_t st;
    int rc[2];
};

int main()
{
    uint8_t *x;
    uint16_t *w;
    float *s_w;
    int8_t *q;
    std::vector<Call> c(T + 1);
    if (cudaMalloc(&x, M * K) || cudaMalloc(&w, N * K * 2) || cudaMalloc(&s_w, N * 4) || cudaMalloc(&q, L * 64)) return 2;
    cudaMemset(x, 0x55, M * K);
    cudaMemset(w, 0x3c, N * K * 2);
    cudaMemset(s_w, 0x3c, N * 4);
    cudaMemset(q, 0x11, L * 64);
    const size_t ws = fqvit_linear_workspace_size(M, K);
    for (Call &i : c)
        if (cudaMalloc(&i.y, M * N) || cudaMalloc(&i.logits, L * LD) || cudaMalloc(&i.ws, ws) || cudaStreamCreate(&i.st))
            return 2;
    cudaDeviceSynchronize();
    auto call = [&](Call &i) {
        i.rc[0] = fqvit_linear_q(x, M, K, K, 128, 0.02f, w, N, s_w, nullptr, 0.05f, 128, i.y, N, nullptr, 0, i.ws, ws, i.st);
        i.rc[1] = fqvit_qk_logits(q, 64, 0, q, 64, 0, 1, L, 64, 0.03f, 0.03f, 0.05f, 0, i.logits, LD, i.st);
    };
    std::atomic<int> ready{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < T; ++t)
        threads.emplace_back([&, t] {
            cudaSetDevice(0);
            cudaFree(nullptr);
            ++ready;
            while (ready.load() < T) {
            }
            call(c[t]);
        });
    for (auto &t : threads) t.join();
    call(c[T]);
    if (cudaDeviceSynchronize()) return 3;
    std::vector<uint8_t> a(M * N), b(M * N), la(L * LD), lb(L * LD);
    cudaMemcpy(b.data(), c[T].y, M * N, cudaMemcpyDeviceToHost);
    cudaMemcpy(lb.data(), c[T].logits, L * LD, cudaMemcpyDeviceToHost);
    int bad = 0;
    for (Call &i : c) {
        if (i.rc[0] || i.rc[1]) {
            ++bad;
            continue;
        }
        cudaMemcpy(a.data(), i.y, M * N, cudaMemcpyDeviceToHost);
        cudaMemcpy(la.data(), i.logits, L * LD, cudaMemcpyDeviceToHost);
        bad += a != b || la != lb;
    }
    printf("%d\n", bad);
    return bad != 0;
}
"""


def test_first_calls_of_many_threads(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = fbuild.build()
    src, exe = tmp_path / "first_calls.cu", tmp_path / "first_calls"
    src.write_text(_PROGRAM)
    subprocess.run([fbuild.nvcc(), *fbuild.ARCH, "-std=c++17", f"-I{fbuild.INCLUDE}", str(src), "-o", str(exe),
                    str(lib), "-Xcompiler", "-pthread"], check=True)
    env = dict(os.environ, LD_LIBRARY_PATH=f"{Path(lib).parent}:{os.environ.get('LD_LIBRARY_PATH', '')}")
    results = [subprocess.run([str(exe)], env=env, capture_output=True, text=True, timeout=120) for _ in range(12)]
    assert [r.returncode for r in results] == [0] * 12, [r.stdout + r.stderr for r in results]
