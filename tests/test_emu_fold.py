"""The integer folded from the four exact digit-product levels
(csrc/emu_arith.cuh, compiled for the host): ((x0 256 + x1) 256 + x2) 256 + x3
for FP32 integers up to each level's bound, the bounds themselves among them."""
import ctypes
import os
import random
import subprocess

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1907_05420_gb300", "csrc")


def test_fold_is_exact(tmp_path):
    cpp, lib = str(tmp_path / "fold.cpp"), str(tmp_path / "fold.so")
    with open(cpp, "w") as f:
        f.write('#include "emu_arith.cuh"\nextern "C" long long fold(float a, float b, float c, float d) '
                "{ return kkt::fold_level2(kkt::fold_level1(kkt::small_f2i(a), b), c) + kkt::exact_f2i(d); }\n")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", SRC, "-o", lib, cpp], check=True)
    fold = ctypes.CDLL(lib).fold
    fold.argtypes = [ctypes.c_float] * 4
    fold.restype = ctypes.c_longlong
    rng = random.Random(4)
    bounds = [2 ** 22, 2 ** 23, 2 ** 24, 2 ** 24]
    draws = [[rng.choice([-b, -b + 1, -1, 0, 1, b - 1, b]) for b in bounds] for _ in range(500)]
    draws += [[rng.randint(-b, b) for b in bounds] for _ in range(5000)]
    for x in draws:
        assert fold(*x) == ((x[0] * 256 + x[1]) * 256 + x[2]) * 256 + x[3], x
