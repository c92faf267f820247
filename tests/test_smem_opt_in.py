"""The opt-in to more than 48 KB of shared memory holds per kernel and device: on the host, with the two CUDA
calls replaced by ones that record what they are asked for."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2401_06132_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

MAIN = r"""
#include "fr_smem.h"
#include <cstdio>
static int dev = 0, sets = 0;
static bool broken = false;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = dev; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute, int bytes)
{
    std::printf("%s %d %d\n", *(const char *)f == 'a' ? "a" : "b", dev, bytes);
    sets++;
    return broken ? cudaErrorInvalidValue : cudaSuccess;
}
int main()
{
    static const char a = 'a', b = 'b';
    static SmemOptIn oa, ob;
    for (int pass = 0; pass < 2; pass++)
        for (dev = 0; dev < 3; dev++) { oa(&a, 60000); ob(&b, 50000); }
    dev = 5; broken = true; oa(&a, 60000); broken = false; oa(&a, 60000); oa(&a, 60000);   // asked again after a failure
    dev = 70; oa(&a, 60000); oa(&a, 60000);                                                // not remembered
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.isdir(CUDA), reason="needs g++ and the CUDA headers")
def test_every_device_is_asked_once(tmp_path):
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text(MAIN)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, "-I", CUDA, str(src), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")[:-1]
    assert out == [f"{k} {d} {n}" for d in range(3) for k, n in (("a", 60000), ("b", 50000))] + ["a 5 60000"] * 2 + ["a 70 60000"] * 2


def test_launches_opt_in_per_device():
    """No launch keeps a process-wide flag of its own for the attribute (the merged launch sets it on every
    call)."""
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        for m in re.finditer(r"cudaFuncSetAttribute\((\w+)", text):
            assert name == "fr_smem.h" or m.group(1) == "k_multi_B", (name, m.group(0))
