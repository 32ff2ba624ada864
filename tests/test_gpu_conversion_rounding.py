"""Caller layout to device layout and back: the deviation D = F - R and the sum F = D + R, R = w_i w_j,
are rounded once, also near rest, where F and R nearly cancel."""
import struct
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1708_05944_gb300 import vlb  # noqa: E402


def rounded(x, dtype):
    """The Fraction x in binary32 or binary64, to nearest even (no underflow here)."""
    bits = 24 if dtype == np.float32 else 53
    if x == 0:
        return dtype(0)
    a = abs(x)
    e = a.numerator.bit_length() - a.denominator.bit_length()
    e -= Fraction(2) ** e > a
    n = a / Fraction(2) ** (e - bits + 1)
    f, r = divmod(n.numerator, n.denominator)
    f += 2 * r > n.denominator or (2 * r == n.denominator and f & 1)
    return dtype(float((1 if x > 0 else -1) * f) * 2.0 ** (e - bits + 1))


def saved_deviation(c, path, n_inst):
    """The device rows of a saved context: (cells, Vp, 2)."""
    c.save(str(path))
    raw = path.read_bytes()
    off = struct.calcsize("=8s6i4i2q") + 4 * n_inst
    d = np.frombuffer(raw[off:], dtype=c.dtype)
    return d.reshape(c.total_cells, -1, 2)


@pytest.mark.parametrize("prec,dtype", [(vlb.VLB_FP64, np.float64), (vlb.VLB_FP32_BULK, np.float32)])
@pytest.mark.parametrize("spec", ["HH(3;4)xH(3;4)", "H(4;5)xH(4;5)", "HH(4;8)xH(4;12)"])
def test_conversion_rounds_once(prec, dtype, spec, tmp_path):
    c = vlb.Couette(spec, prec, [dict(n_cells=4, r_in=1.0, r_out=2.0)], [(0.1, 1.0)], [(0.0, 1.0)], [0.1], [1])
    w0, w1 = (vlb.vlb_quadrature(c.model, a)[1] for a in (0, 1))
    R = [[Fraction(float(a)) * Fraction(float(b)) for b in w1] for a in w0]
    rng = np.random.default_rng(61)
    F = np.empty(c.f_shape(), dtype=dtype)
    base = np.outer(w0, w1)
    F[0] = base                                                # at rest to rounding
    F[1] = base * (1.0 + 1e-7 * rng.uniform(-1, 1, F[1].shape))  # a few units in the last place away
    F[2] = base * (1.0 + 1e-3 * rng.uniform(-1, 1, F[2].shape))
    F[3] = base * rng.uniform(0.1, 4.0, F[3].shape)
    c.set_f(F)
    D = saved_deviation(c, tmp_path / "state", 1)
    back = c.read_f()
    c.close()
    nq1 = len(w1)
    for cell in range(4):
        for d in range(2):
            for i in range(len(w0)):
                for j in range(nq1):
                    got = D[cell, i * nq1 + j, d]
                    # single precision: R itself is held to 53 bits, and a sum lies that close to a tie once in 2^29
                    r = R[i][j] if dtype == np.float64 else Fraction(float(w0[i]) * float(w1[j]))
                    assert got == rounded(Fraction(float(F[cell, d, i, j])) - r, dtype)
                    assert back[cell, d, i, j] == rounded(Fraction(float(got)) + r, dtype)
