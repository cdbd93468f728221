"""Launchers of the streaming key passes given an element type or a row length that they have no kernel for: an error, and
nothing launched.  (The entry points refuse both before; compiled and run without a device.)"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_26678_b200", "csrc")

PROGRAM = r"""
#include "nkv_common.cuh"
#include <stdio.h>
int main() {
    nkv::ScoreParams sp = {};
    sp.window = 64, sp.block = 128, sp.nblocks = 1;
    float* none = nullptr;
    int bad = 0;
    const int forms[][2] = {{99, 128}, {-1, 64}, {NKV_BF16, 96}, {NKV_F16, 32}, {NKV_F32, 256}};
    for (auto& f : forms) {
        const nkv::TensorView K = {nullptr, 0, 0, 1, 100, f[1]};
        int64_t launches = 0;
        const cudaError_t e[3] = {nkv::launch_anchor_sums(K, f[0], 1, sp, none, none, 0, &launches),
                                  nkv::launch_stream_a(K, f[0], 1, sp, none, none, none, nullptr, nullptr, 148, 0, &launches),
                                  nkv::launch_stream_b(K, f[0], 1, sp, none, none, none, none, none, none, nullptr, nullptr, 148, 0, &launches)};
        for (int i = 0; i < 3; ++i)
            if (e[i] != cudaErrorInvalidValue || launches != 0) {
                printf("launcher %d, type %d, d = %d: %s, %d launches\n", i, f[0], f[1], cudaGetErrorName(e[i]), (int)launches);
                ++bad;
            }
    }
    return bad;
}
"""


def test_a_form_without_a_kernel_is_an_error(tmp_path):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if not (os.path.exists(nvcc) or shutil.which(nvcc)):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "forms.cu", tmp_path / "forms"
    src.write_text(PROGRAM)
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                           str(src), os.path.join(CSRC, "nkv_stream.cu"), "-o", str(exe)])
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")   # nothing may be launched
    done = subprocess.run([str(exe)], capture_output=True, text=True, env=env)
    assert done.returncode == 0, done.stdout
