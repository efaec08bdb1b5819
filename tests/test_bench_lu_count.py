"""bench.py's count of the kernels behind the mixed path's G and T^-1 update (no
GPU): the blocked LU is LU (1/3) and two triangular solves with M right-hand sides
(1), 4/3 M^3 complex multiply-adds of 8 flop, six bf16 products each against the
bf16 rate; the T^-1 update is 1/2 M^3 complex multiply-adds as 36 digit products
from M = 100 up, 48 FP32 instructions below, and FP64 outside the mixed path."""
import importlib

import pytest


def test_blocked_lu_and_tinv_counts():
    bench = importlib.import_module("bench")
    bf16 = bench.PEAKS.get("bf16_tflops", 1900.0)
    M, W = 257, 1024
    r = bench.roofline({"green": {"ms": 36.0, "n_timed": 5}}, M, W, "mixed", green_tc="lu")
    macs = 4.0 / 3.0 * M ** 3 * W
    assert r["bound"] == "tensor" and r["peak"] == bf16 and r["traffic"] is None
    assert r["achieved"] == pytest.approx(6 * 8 * macs / (36.0 / 5 / 1e3) / 1e12)
    assert bench.kernel_model("tinv", 123, 1, "mixed")[:3] == (36 * 8 * 0.5 * 123 ** 3, "tensor", bf16)
    assert bench.kernel_model("tinv", 57, 1, "mixed")[:3] == (2 * 48 * 0.5 * 57 ** 3, "alu", bench.FP32_PEAK_TFLOPS)
    assert bench.kernel_model("tinv", 123, 1, "fp64")[:3] == (8 * 0.5 * 123 ** 3, "alu", bench.FP64_PEAK_TFLOPS)
