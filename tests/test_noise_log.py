"""The gradient noise's -2 ln u (minus_2_ln in device.cuh), restated in numpy
with the coefficients read from the source: every u = k 2^-24, k = 1 .. 2^24,
against float64.  The source states these figures."""
import os
import re

import numpy as np

from paper_2110_04175_gb300 import build as rs_build


def _coefficients() -> list:
    with open(os.path.join(rs_build.CSRC, "device.cuh")) as f:
        text = f.read()
    body = text[text.index("Pair minus_2_ln(Pair u)"):]
    body = body[:body.index("\n}")]
    first = re.search(r"Pair p = pack\((\S+)f\);", body)
    rest = re.findall(r"p = fma2\(p, f, pack\((\S+)f\)\);", body)
    assert "fma2(pack(__int2float_rn(e0), __int2float_rn(e1)), c, mul2(f, p))" in body  # as restated below
    return [np.float32(v) for v in [first.group(1), *rest]]  # highest degree first


def _fma(a, b, c):
    # the product of two fp32 values is exact in fp64
    return (np.float64(a) * np.float64(b) + np.float64(c)).astype(np.float32)


def _minus_2_ln(u: np.ndarray, coef: list) -> np.ndarray:
    bits = u.view(np.int32)
    e = (bits - np.int32(0x3F3504F3)) & np.int32(-(1 << 23))
    f = (bits - e).view(np.float32) - np.float32(1)
    p = np.full_like(f, coef[0])
    for c in coef[1:]:
        p = _fma(p, f, c)
    return _fma(e.astype(np.float32), np.float32(-2 * np.log(2) * 2.0 ** -23), f * p)


def test_radius_over_every_uniform():
    coef = _coefficients()
    assert len(coef) == 9 and coef[-1] == -2
    worst = worst_rel = squares = 0.0
    for lo in range(1, (1 << 24) + 1, 1 << 21):
        k = np.arange(lo, lo + (1 << 21), dtype=np.float32)
        u = k * np.float32(2.0 ** -24)
        got = _minus_2_ln(u, coef).astype(np.float64)
        want = -2 * np.log(u.astype(np.float64))
        assert got.min() >= 0
        nz = want > 0
        worst_rel = max(worst_rel, float(np.max(np.abs(got[nz] - want[nz]) / want[nz])))
        assert np.all(got[~nz] == 0)
        err = np.abs(np.sqrt(got) - np.sqrt(want))
        worst = max(worst, float(err.max()))
        squares += float(np.sum(err ** 2))
    assert worst <= 1.4e-7 and worst_rel <= 2.0e-7
    assert np.sqrt(squares / (1 << 24)) <= 2.2e-8
