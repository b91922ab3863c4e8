"""What the launchers keep per device, compiled for the host against fakes of the CUDA calls: on a
process's second device a kernel gets its shared-memory attribute again and the SM count is
that device's; on a device that was seen before neither is asked for again; a failed call is not
remembered; without a device the SM count is the host-only default."""
import os
import shutil
import subprocess

import pytest

from paper_2506_02965_gb300 import build as B

PROGRAM = r"""
#include "device_state.h"
#include <cstdio>
static int dev = 0, sets = 0, asks = 0;
static bool fail_set = false;
extern "C" cudaError_t CUDARTAPI cudaGetDevice(int* d) { *d = dev; return dev < 0 ? cudaErrorNoDevice : cudaSuccess; }
extern "C" cudaError_t CUDARTAPI cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int d) { ++asks; *v = 100 + d; return cudaSuccess; }
extern "C" cudaError_t CUDARTAPI cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) {
    ++sets;
    return fail_set ? cudaErrorInvalidValue : cudaSuccess;
}
void k1(int) {}
void k2(int) {}
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
int main() {
    using namespace moe;
    CHECK(sm_count() == 100 && sm_count() == 100 && asks == 1);
    CHECK(allow_dynamic_smem<k1>(1) == cudaSuccess && allow_dynamic_smem<k1>(1) == cudaSuccess && sets == 1);
    CHECK(allow_dynamic_smem<k2>(1) == cudaSuccess && sets == 2);
    dev = 3;
    CHECK(sm_count() == 103 && asks == 2);
    CHECK(allow_dynamic_smem<k1>(1) == cudaSuccess && sets == 3);
    dev = 0;
    CHECK(sm_count() == 100 && asks == 2);
    CHECK(allow_dynamic_smem<k1>(1) == cudaSuccess && sets == 3);
    dev = 5;
    fail_set = true;
    CHECK(allow_dynamic_smem<k1>(1) == cudaErrorInvalidValue && sets == 4);
    fail_set = false;
    CHECK(allow_dynamic_smem<k1>(1) == cudaSuccess && sets == 5);
    dev = 1000;
    CHECK(sm_count() == 1100 && allow_dynamic_smem<k1>(1) == cudaSuccess && allow_dynamic_smem<k1>(1) == cudaSuccess && sets == 7);
    dev = -1;
    CHECK(sm_count() == 148);
    return 0;
}
"""


def test_state_is_kept_per_device(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("needs g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    r = subprocess.run([gxx, "-std=c++17", "-I", B.CSRC, "-I", cuda, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
