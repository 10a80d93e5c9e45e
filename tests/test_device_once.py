"""The opt-ins to large dynamic shared memory are made on every device that a process
uses, once each: the C++ of csrc/tk_device_once.h against a stand-in for the CUDA
runtime."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1010_3816_gb300", "csrc")

RUNTIME = """
#pragma once
#include <stddef.h>
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1 };
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize };
extern int device, sets[3], refuse;
inline cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
inline cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int bytes)
{
    if (refuse || bytes != 51328) return cudaErrorInvalidValue;
    sets[device == 100 ? 2 : device]++;
    return cudaSuccess;
}
"""

MAIN = """
#include "tk_device_once.h"
#include <stdio.h>
#include <initializer_list>
int device, sets[3], refuse;
static cudaError_t launch()   // as a launcher does before each launch
{
    static tk::DeviceOnce once;
    return tk::allow_smem(once, (const void *)launch, 51328);
}
int main()
{
    refuse = 1;
    int bad = launch() != cudaErrorInvalidValue;      // a failure is not remembered
    refuse = 0;
    for (int d : {0, 1, 0, 1, 0, 100, 100}) {
        device = d;
        bad += launch() != cudaSuccess;
    }
    printf("%d %d %d %d\\n", bad, sets[0], sets[1], sets[2]);
}
"""


def test_each_device_once(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "main.cc").write_text(MAIN)
    exe = str(tmp_path / "once")
    subprocess.run(["g++", "-std=c++17", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "main.cc"), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split() == ["0", "1", "1", "2"]


def test_no_function_attribute_is_set_once_per_process():
    """Every opt-in goes through allow_smem, or is made at each call."""
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            text = open(os.path.join(CSRC, name)).read()
            assert not re.search(r"static[^;]*=\s*cudaFuncSetAttribute", text), name
