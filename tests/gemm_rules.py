"""The host rules of the GEMMs (csrc/dsq_gemm8_rule.h, for a GPU of 148 SMs) compiled for the tests."""
import ctypes as C
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


class Rules:
    def __init__(self, so):
        lib = self.lib = C.CDLL(so)
        lib.tile.restype = C.c_double
        lib.tile.argtypes = [C.c_int64] * 3 + [C.c_int] + [C.POINTER(C.c_int)] * 2
        lib.two_passes.argtypes = [C.c_int64] * 3 + [C.c_int] * 2 + [C.c_double]
        lib.wgemm_form.argtypes = [C.c_int64] * 3 + [C.c_double]
        lib.gemm_small.argtypes = [C.c_int64] * 3 + [C.c_int] * 2 + [C.POINTER(C.c_int)] * 2
        lib.gemm_form.argtypes = [C.c_int64] * 3 + [C.c_int] * 2 + [C.c_double, C.c_int]

    def tile(self, operands, m, n, k):
        """((width, parts of K), clocks) of the second pass."""
        bn, split = C.c_int(), C.c_int()
        kblocks = -(-k // {"i8": 128, "bf16": 64, "f4": 256}[operands])
        clocks = self.lib.tile(m, n, kblocks, 240 if operands == "f4" else 256, C.byref(bn), C.byref(split))
        return (bn.value, split.value), clocks

    def gemm_form(self, m, n, k, bits, outs, room):
        """Of dsq_gemm with `outs` arrays written: "fused", "two" passes or "small"."""
        _, clocks = self.tile("i8" if bits == 4 else "f4", m, n, k)
        return ("fused", "two", "small")[self.lib.gemm_form(m, n, k, bits, outs, clocks, room)]

    def two_passes(self, m, n, k, bits, f4, clocks):
        return self.lib.two_passes(m, n, k, bits, f4, clocks)

    def gemm_small(self, m, n, k, bits, outs):
        """(rows, warps) of a block of the little-work kernel."""
        rows, warps = C.c_int(), C.c_int()
        self.lib.gemm_small(m, n, k, bits, outs, C.byref(rows), C.byref(warps))
        return rows.value, warps.value

    def wgemm_form(self, m, n, k):
        """Of a weight-only GEMM of more than 32 rows: columns of a block of the kernel of few rows, 0: two passes."""
        return self.lib.wgemm_form(m, n, k, self.tile("bf16", m, n, k)[1])


@pytest.fixture(scope="session")
def rules(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("rules") / "gemm_rules_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", os.path.join(HERE, "gemm_rules_host.cpp"), "-o", so],
                   check=True)
    return Rules(so)
