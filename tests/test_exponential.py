"""The exponential that the query stage takes on the FMA pipe, its arithmetic done over in numpy with the constants of the source."""
import os
import re

import numpy as np

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24899_b200", "csrc", "tensor_qpass.cu")


def _fma(a, b, c):
    return (a.astype(np.float64) * np.float64(b) + np.float64(c)).astype(np.float32) if np.isscalar(b) else \
        (a.astype(np.float64) * b.astype(np.float64) + np.float64(c)).astype(np.float32)


def _ex2_fma(x):
    with open(SOURCE) as f:
        body = re.search(r"AS_DEV float2 ex2_fma\(float2 x\) \{(.*?)\n\}", f.read(), re.S).group(1)
    least = [np.float32(v) for v in re.findall(r"fmax_nan\(x\.[xy], (-?[0-9.]+)f\)", body)]
    c = [np.float32(v) for v in re.findall(r"both\((-?[0-9.e+-]+)f\)", body)]
    magic, coeff = c[0], c[3:]
    assert c[1] == -magic and c[2] == -1 and len(coeff) == 6 and coeff[-1] == 1 and len(least) == 2 and least[0] == least[1]
    x = np.maximum(x, least[0])                              # (a NaN stays)
    n = ((x + magic).astype(np.float32) - magic).astype(np.float32)
    f = (x - n).astype(np.float32)
    assert not (np.abs(f) > 0.5).any()
    y = np.full_like(f, coeff[0])
    for k in coeff[1:]:
        y = _fma(y, f, k)
    bits = ((x + magic).astype(np.float32).view(np.uint32) << np.uint32(23)) + np.uint32(0x3f800000)
    got = (y * bits.view(np.float32)).astype(np.float32)
    if "fmul2_ftz(y, p)" in body:
        got[np.abs(got) < np.finfo(np.float32).tiny] = 0
    return got


def test_within_the_error_of_the_special_function_unit():
    """ex2.approx.ftz.f32 is documented to 2^-22 = 2.4e-7 relative; the polynomial's 1.08e-7 and a rounding or two stay below that."""
    x = np.concatenate([np.linspace(-126, 8, 2000003), np.linspace(-1, 1, 500001), np.linspace(0.5, 0.501, 200001), np.arange(-126, 9)]).astype(np.float32)
    got, want = _ex2_fma(x), np.exp2(x.astype(np.float64))
    inside = want >= 2.0 ** -126 * (1 + 2.0 ** -22)          # (at the very end of the range a rounding decides what is flushed)
    assert float(np.abs(got / want - 1)[inside].max()) <= 1.72e-7
    assert got[x == 0.0][0] == 1.0


def test_nothing_is_left_below_the_normal_range():
    x = np.concatenate([-126 - np.logspace(-5, 6, 20001), [-126.25, -126.5, -127, -127.5, -128, -1e30, -np.inf]]).astype(np.float32)
    x = x[x < -126]
    assert not _ex2_fma(x).any()
    assert np.isnan(_ex2_fma(np.array([np.nan], np.float32))).all()
