"""The integer bounds on the fixed-point phi that the phase march tests before the interfacial gate
q = phi (1 - phi) >= q_th (Eq. 58, evaluated in binary32 as the kernels evaluate it): every value that
passes the gate lies within the bounds, at both edges and for thresholds up to the largest possible q,
where the slope of q vanishes and one rounding of q moves the edge by 1.5e-4; and the bounds are not
wider than the rounding of q asks for. csrc/gate_bounds.h is compiled here for the host."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_17481_gb300", "csrc")
F32 = np.float32


@pytest.fixture(scope="module")
def bounds(tmp_path_factory):
    d = tmp_path_factory.mktemp("gate")
    src, lib = d / "g.cpp", d / "g.so"
    src.write_text('#include "gate_bounds.h"\n'
                   'extern "C" void bounds(float q, int32_t *lo, uint32_t *span) { lbm::gate_bounds(q, *lo, *span); }\n')
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    L = ctypes.CDLL(str(lib))

    def f(q_th):
        lo, span = ctypes.c_int32(), ctypes.c_uint32()
        L.bounds(ctypes.c_float(q_th), ctypes.byref(lo), ctypes.byref(span))
        return lo.value, span.value
    return f


def _q(v):
    """q of the fixed-point values as the kernels evaluate it, every operation rounded to binary32."""
    pc = np.clip(v.astype(np.int32).astype(F32) * F32(2.0 ** -30), F32(0), F32(1))
    return pc * (F32(1) - pc)


def _values(q_th):
    """Fixed-point values: 400,000 around each edge, the whole range of int32 in steps, and its ends."""
    root = 0.5 * (1.0 - np.sqrt(max(0.0, 1.0 - 4.0 * q_th)))
    near = np.arange(-400_000, 400_000, dtype=np.int64)
    v = np.concatenate([near + int(root * 2 ** 30), near + int((1 - root) * 2 ** 30), near,
                        np.arange(-2 ** 31, 2 ** 31, 7919, dtype=np.int64), [-2 ** 31, 2 ** 31 - 1]])
    return v[(v >= -2 ** 31) & (v < 2 ** 31)]


@pytest.mark.parametrize("q_th", [1e-50, 1e-40, 1e-12, 1e-8, 1e-6, 0.01, 0.07, 0.125, 0.2, 0.2499, 0.24999, 0.249999,
                                  0.25 - 6e-7, 0.2499999, 0.25 - 1e-8, 0.25])
def test_every_value_the_gate_passes_is_within_the_bounds(bounds, q_th):
    lo, span = bounds(q_th)
    v, th = _values(q_th), F32(q_th)
    q = _q(v)
    passes = ((v - lo) & 0xFFFFFFFF) <= span  # the march's unsigned comparison
    gated = q >= th
    assert gated.any()
    assert not np.any(gated & ~passes)
    # three roundings of at most 2^-25 each and the march's own margin: nothing further out is let through
    if th > 0:
        assert not np.any(passes & (q < th - F32(3e-7)))
