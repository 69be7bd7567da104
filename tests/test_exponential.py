"""The exponential that the query stage takes on the FMA pipe, its arithmetic done over in numpy with the constants of the source."""
import os
import re

import numpy as np

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24899_b200", "csrc", "tensor_qpass.cu")


def _fma(a, b, c):
    return (a.astype(np.float64) * np.float64(b) + np.float64(c)).astype(np.float32) if np.isscalar(b) else \
        (a.astype(np.float64) * b.astype(np.float64) + np.float64(c)).astype(np.float32)


def test_within_the_error_of_the_special_function_unit():
    """ex2.approx.ftz.f32 is documented to 2^-22 relative; the polynomial's 9.1e-8 and a rounding or two stay below that."""
    with open(SOURCE) as f:
        body = re.search(r"AS_DEV float2 ex2_fma\(float2 x\) \{(.*?)\n\}", f.read(), re.S).group(1)
    c = [np.float32(v) for v in re.findall(r"both\((-?[0-9.e+-]+)f\)", body)]
    magic, coeff = c[0], c[3:]
    assert c[1] == -magic and c[2] == -1 and len(coeff) == 6 and coeff[-1] == 1
    x = np.concatenate([np.linspace(-126, 8, 2000003), np.linspace(-1, 1, 500001), np.arange(-126, 9)]).astype(np.float32)
    n = ((x + magic).astype(np.float32) - magic).astype(np.float32)
    f = (x - n).astype(np.float32)
    assert float(np.abs(f).max()) <= 0.5
    y = np.full_like(f, coeff[0])
    for k in coeff[1:]:
        y = _fma(y, f, k)
    bits = ((x + magic).astype(np.float32).view(np.uint32) << np.uint32(23)) + np.uint32(0x3f800000)
    got = (y * bits.view(np.float32)).astype(np.float32)
    want = np.exp2(x.astype(np.float64))
    assert float(np.abs(got / want - 1).max()) <= 2.0 ** -22
    assert got[x == 0.0][0] == 1.0
