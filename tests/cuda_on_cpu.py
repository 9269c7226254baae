"""Compiles a kernel's source file for the CPU (cuda_on_cpu.h): `extern
__shared__` arrays, launches and inline PTX are replaced in a copy of the
sources, everything else is the file as it stands."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(ROOT, "paper_2602_17335_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

PTX = [("mbarrier.try_wait", "ok = 1;"), ("cp.async.bulk.shared", "memcpy(dst, src, bytes);"),
       ("ld.global.v4.u32", "v = *p;"), ("ld.global.u8", "v = *p;"), ("ld.shared.u32", "memcpy(&v, emu::smem + a, 4);"),
       ("mbarrier.", ";"), ("fence.", ";"), ("prefetch.", ";")]


def _replace_ptx(text):
    out, at = [], 0
    while True:
        k = text.find("asm volatile(", at)
        if k < 0:
            return "".join(out) + text[at:]
        out.append(text[at:k])
        j, depth, quoted = k + len("asm volatile("), 1, False
        while depth:
            c = text[j]
            if c == '"' and text[j - 1] != "\\":
                quoted = not quoted
            elif not quoted:
                depth += (c == "(") - (c == ")")
            j += 1
        j = text.index(";", j) + 1
        body = text[k:j]
        out.append(next((new for name, new in PTX if name in body), body))
        out[-1] += "\n" * body.count("\n")
        at = j


def translate(text):
    text = _replace_ptx(text)
    text = re.sub(r"extern __shared__ __align__\(\d+\) uint8_t (\w+)\[\];", r"uint8_t* const \1 = emu::smem;", text)
    return re.sub(r"(\b[\w]+(?:<[\w, ]+>)?)<<<(.*?), (\w+|\(.*?\)), ([^,]+), s>>>\((.*?)\);",
                  r"emu::launch([=] { \1(\5); }, \2, \3, \4);", text, flags=re.S)


def compile_kernels(tmp, harness, sanitize):
    """The library of `harness` (which includes the kernel sources), or a skip."""
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("no g++ or CUDA headers")
    src = os.path.join(str(tmp), "csrc")
    os.makedirs(src, exist_ok=True)
    for f in os.listdir(CSRC):
        if f.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(CSRC, f)) as a, open(os.path.join(src, f), "w") as b:
                b.write(translate(a.read()))
    inc = ["-I", src, "-I", HERE, "-I", os.path.join(ROOT, "include"), "-I", CUDA_INC]
    base = ["g++", "-std=c++17", "-fPIC", "-w", *inc]
    fib, lib = os.path.join(str(tmp), "fibers.o"), os.path.join(str(tmp), "kernels.so")
    subprocess.run([*base, "-O2", "-U_FORTIFY_SOURCE", "-c", os.path.join(HERE, "cuda_on_cpu.cpp"), "-o", fib], check=True)
    san = ["-fsanitize=address,bounds,alignment,shift", "-fno-omit-frame-pointer", "--param", "asan-stack=0"] if sanitize else []
    subprocess.run([*base, "-O1", "-g", *san, "-shared", os.path.join(HERE, harness), fib, "-o", lib], check=True)
    return lib
