"""The row scale of the emulated-FP64 operands: the exponent found from the
bits of the largest magnitude (csrc/emu_arith.cuh, compiled for the host)
against Python's frexp, which returns m in [0.5, 1) and e with v = m 2^e."""
import ctypes
import math
import os
import random
import struct
import subprocess

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1907_05420_gb300", "csrc")


def test_scale_exponent_is_frexp(tmp_path):
    cpp, lib = str(tmp_path / "scale.cpp"), str(tmp_path / "scale.so")
    with open(cpp, "w") as f:
        f.write('#include "emu_arith.cuh"\nextern "C" int scale(double v) '
                "{ return kkt::scale_exponent(kkt::magnitude_bits(v)); }\n")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", SRC, "-o", lib, cpp], check=True)
    scale = ctypes.CDLL(lib).scale
    scale.argtypes = [ctypes.c_double]
    rng = random.Random(3)
    vals = [0.0, -0.0, 1.0, 5e-324, 2.2250738585072014e-308, 2.225073858507201e-308, 1.7976931348623157e308]
    vals += [struct.unpack("d", struct.pack("Q", rng.getrandbits(63) % (2047 << 52)))[0] for _ in range(2000)]
    for v in vals:
        for s in (v, -v):
            assert scale(s) == (math.frexp(v)[1] if v else 0), v
