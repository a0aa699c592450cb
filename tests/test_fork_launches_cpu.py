"""Launches on two streams (csrc/fork_launches.h) against a recorder in place of the CUDA runtime: whatever
launch fails, the second stream is behind the first one's earlier work and joins it again."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#pragma once
#include <cstring>
enum cudaError_t { cudaSuccess = 0 };
typedef int cudaStream_t;
typedef int cudaEvent_t;
extern char log_[256];
inline void note(char op, int arg) { const char s[3] = {op, (char)('0' + arg), 0}; strcat(log_, s); }
inline cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t s) { note('r', s); return cudaSuccess; }
inline cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, int) { note('w', s); return cudaSuccess; }
"""

SRC = r"""
#include "fork_launches.h"
char log_[256];
extern "C" int run(int n, int failing, char* out) {
    log_[0] = 0;
    const int e = mcao::fork_launches(0, 1, 7, n, [&](int i, cudaStream_t s) {
        if (i == failing) return (cudaError_t)5;
        note('l', s);
        return cudaSuccess;
    });
    strcpy(out, log_);
    return e;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("fork")
    (d / "cuda_runtime.h").write_text(FAKE)
    (d / "fork.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", str(d), "-I", os.path.join(ROOT, "paper_1608_00386_gb300", "csrc"),
                    str(d / "fork.cpp"), "-o", str(d / "fork.so")], check=True)
    f = ctypes.CDLL(str(d / "fork.so")).run

    def call(n, failing):
        buf = ctypes.create_string_buffer(256)
        return f(n, failing, buf), buf.value.decode()
    return call


@pytest.mark.parametrize("n", range(5))
@pytest.mark.parametrize("failing", range(-1, 4))
def test_the_second_stream_always_joins(run, n, failing):
    e, log = run(n, failing)
    fails = 0 <= failing < n
    assert e == (5 if fails else 0)
    launches = "".join("l0" if i == 0 else "l1" for i in range(failing if fails else n))
    assert log == (launches if n < 2 else "r0w1" + launches + "r1w0")
