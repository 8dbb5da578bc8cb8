"""The weight quantizer's multiplication rule, restated on the CPU: a row whose few bf16 values next to the half-integers
(k + 1/2) s give the same code by one multiply-add (with 1 / s or a neighbour of it) and by an IEEE division gives the same code
everywhere."""
import numpy as np
import pytest

MAGIC = 12582912.0


def code_div(w, s):
    return np.clip(np.rint((w / s).astype(np.float32)), -8, 7).astype(int)


def code_mul(w, r):  # float64 holds the product and the sum of the fused multiply-add
    f = (w.astype(np.float64) * np.float64(r) + MAGIC).astype(np.float32)
    c = f.view(np.uint32) & 15
    return np.where(c > 7, c.astype(int) - 16, c.astype(int))


@pytest.mark.parametrize("exponent", [1, 60, 120, 127, 200, 253])
def test_rows_that_pass_the_check_agree_with_the_division_everywhere(exponent):
    checked = 0
    for mantissa in range(128):
        top = (exponent << 7) | mantissa
        mx = np.array([top << 16], np.uint32).view(np.float32)[0]
        s = np.float32(mx) / np.float32(7.0)
        if not 1e-30 < s < 1e30:
            continue
        near = []
        for k in range(7):
            h = int(np.array([np.float32(k + 0.5) * s], np.float32).view(np.uint32)[0]) >> 16
            near += [h + d for d in (-1, 0, 1, 2)]
        b = (np.array(near, np.uint32) << 16).view(np.float32)
        one = np.float32(1.0) / s
        agree = [r for r in (one, np.nextafter(one, np.float32(np.inf)), np.nextafter(one, np.float32(0))) if np.array_equal(code_mul(b, r), code_div(b, s))]
        checked += bool(agree)
        w = (np.arange(0, top + 1, dtype=np.uint32) << 16).view(np.float32)
        w = np.concatenate([w, -w])
        for r in agree:
            assert np.array_equal(code_mul(w, r), code_div(w, s)), (exponent, mantissa)
    assert checked > 100 or exponent in (1, 253)
