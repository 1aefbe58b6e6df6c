"""The shared-memory allowance of a kernel (csrc/smem_limit.h) belongs to a device: a process that uses several asks once on
each, and a refusal on one is neither kept nor taken for the others. Compiled here with g++ against stand-ins of the
two runtime calls; and the launchers that take more than 48 KB ask through it."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2303_15861_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

HARNESS = r"""
#include "smem_limit.h"
#include <cstdio>
static int device = 0, calls = 0;
static bool refuse = false;
extern "C" cudaError_t CUDARTAPI cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t CUDARTAPI cudaFuncSetAttribute(const void*, enum cudaFuncAttribute, int) {
    ++calls;
    return refuse ? cudaErrorInvalidValue : cudaSuccess;
}
int main() {
    adr::SmemLimit one, other;
    const void* k = &calls;
    auto ask = [&](adr::SmemLimit& l, int dev, bool no) {
        device = dev;
        refuse = no;
        const int before = calls;
        const cudaError_t e = l.allow(k, 200000);
        std::printf("%d%s ", calls - before, e == cudaSuccess ? "" : "!");
    };
    ask(one, 0, false); ask(one, 0, false);                    // first and later launches
    ask(one, 3, false); ask(one, 3, false); ask(one, 0, false);  // another device
    ask(one, 5, true);  ask(one, 5, false); ask(one, 5, false);  // refused once
    ask(one, 70, false); ask(one, 70, false);                  // beyond the 64 that are remembered
    ask(other, 0, false);                                      // another kernel
    return 0;
}
"""


def test_allowed_once_on_every_device(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-std=c++17", "-O1", f"-I{CSRC}", f"-I{CUDA_INC}", str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["1", "0", "1", "0", "0", "1!", "1", "0", "1", "1", "1"]


@pytest.mark.parametrize("name", ["contract_f64.cu", "contract_simt.cu", "contract_tc.cu", "batch_tc.cu"])
def test_launchers_ask_through_it(name):
    text = open(os.path.join(CSRC, name)).read()
    assert "cudaFuncSetAttribute" not in text
    assert len(re.findall(r"\bSmemLimit\b", text)) == 1
