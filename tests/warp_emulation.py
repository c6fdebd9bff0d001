"""Device functions of csrc on the CPU: the headers are compiled by g++ with the stand-ins of
warp_emulation.h, their few asm statements replaced by the same operation in C++."""
from __future__ import annotations

import ctypes
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2506_22408_gb300", "csrc")
ASM = [
    (r'asm\("mul\.wide\.s32 %0, %1, %2;" : "=l"\((\w+)\) : "r"\((\w+)\), "r"\((\w+)\)\);', r"\1 = (long long)\2 * \3;"),
    (r'asm\("mad\.wide\.s32 %0, %1, %2, %3;" : "=l"\((\w+)\) : "r"\((\w+)\), "r"\((\w+)\), "l"\((\w+)\)\);',
     r"\1 = (long long)\2 * \3 + \4;"),
    (r'asm\("rcp\.approx\.ftz\.f32 %0, %1;" : "=f"\((\w+)\) : "f"\((.*)\)\);', r"\1 = emu::rcp(\2);"),
    (r'asm volatile\("bar\.sync %0, %1;" ::"r"\(\w+\), "n"\(\w+\) : "memory"\);', "emu::bar();"),
    (r'asm\("cvt\.rn\.bf16x2\.f32 %0, %1, %2;" : "=r"\((\w+)\) : "f"\((\w+)\), "f"\((\w+)\)\);',
     r"\1 = (__float_as_uint(\2) & 0xffff0000u) | (__float_as_uint(\3) >> 16);"),  # exact in BF16
    (r'asm\("mov\.u32 %0, %%dynamic_smem_size;" : "=r"\((\w+)\)\);', r"\1 = 0;"),
]


def cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    for d in (inc, "/usr/local/cuda/include"):
        if os.path.exists(os.path.join(d, "cuda_runtime.h")):
            return d
    pytest.skip("CUDA headers not found")


def host_header(name, dst, edit=None):
    """Copies a header (asm replaced, edit(text) applied) and what it includes into dst."""
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    for pat, rep in ASM:
        text = re.sub(pat, rep, text)
    if edit:
        text = edit(name, text)
    left = re.search(r"\basm\b[^;]*;", text)
    assert left is None, (name, left.group(0))
    with open(os.path.join(dst, name), "w") as f:
        f.write(text)
    for inc in re.findall(r'#include "(qcs_\w+\.\w+)"', text):
        if not os.path.exists(os.path.join(dst, inc)):
            host_header(inc, dst, edit)


def compile_host(source, headers, dst, edit=None):
    """The shared library of a C++ source that includes warp_emulation.h and device headers."""
    for h in headers:
        host_header(h, dst, edit)
    src, lib = os.path.join(dst, "host.cpp"), os.path.join(dst, "libhost.so")
    with open(src, "w") as f:
        f.write('#include "warp_emulation.h"\nemu::Block *emu::blk = nullptr;\n')
        f.write("".join(f'#include "{h}"\n' for h in headers) + source)
    subprocess.run(["g++", "-O1", "-fwrapv", "-fno-strict-aliasing", "-w", "-std=c++17", "-fPIC", "-shared", "-I", dst,
                    "-I", HERE, "-I", os.path.join(ROOT, "include"), "-I", cuda_include(), src, "-o", lib], check=True)
    return ctypes.CDLL(lib)
