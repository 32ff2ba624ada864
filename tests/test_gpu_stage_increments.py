"""What the Shakhov correction adds, held to its own size: at a time step where it is far above the rounding of
the distribution it is added to."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle.couette import CouetteGrid, CouetteOracle, Wall  # noqa: E402
from paper_1708_05944_gb300 import vlb  # noqa: E402
from paper_1708_05944_gb300.inputs import perturbation  # noqa: E402
from tests.helpers import to_lib, to_oracle  # noqa: E402

PRECS = [(vlb.VLB_FP64, np.float64, 2.0 ** -53), (vlb.VLB_FP32_BULK, np.float32, 2.0 ** -24)]


def check(got, ref, top, eps, relative):
    """Increments against the oracle's: four roundings of the distribution (stored and read, on either side of
    the difference) and the roundings of the increment's own terms; the increment has to be fifty times that."""
    tol = 4 * eps * top + relative * np.abs(ref).max()
    assert np.abs(ref).max() > 50 * tol
    assert np.abs(got - ref).max() < tol


# the correction is two dot products of a few projections, some thirty roundings of a term of its size
@pytest.mark.parametrize("prec,dtype,eps", PRECS)
@pytest.mark.parametrize("spec,n", [("HH(4;8)xH(4;12)", 3), ("HH(4;8)xHH(4;10)", 5), ("HH(3;4)xH(3;4)", 3),
                                    ("HH(3;4)xH(3;5)", 4)])
def test_shakhov_term(prec, dtype, eps, spec, n):
    dt = 1e-2
    walls = Wall(0.2, 1.0), Wall(0.0, 1.05)
    oracles = [CouetteOracle(spec, CouetteGrid(n, 1.0, 2.0), *walls, 0.1, 1, prandtl=p) for p in (2.0 / 3.0, None)]
    F = oracles[0].initial_equilibrium()
    F = (F * perturbation(F.shape, seed=91, amplitude=0.03)).astype(dtype).astype(np.float64)
    out = []
    for shakhov in (True, False):
        c = vlb.Couette(spec, prec, [dict(n_cells=n, r_in=1.0, r_out=2.0)], [(0.2, 1.0)], [(0.0, 1.05)], [0.1], [1])
        if shakhov:
            c.set_collision(vlb.VLB_SHAKHOV, 2.0 / 3.0)
        c.set_f(to_lib(F).astype(dtype))
        c.stage(dt, 1)
        out.append(to_oracle(c.read_f()).astype(np.float64))
        c.close()
    ref = [o.stage(1, dt, F, F) for o in oracles]
    check(out[0] - out[1], ref[0] - ref[1], np.abs(ref[1]).max(), eps, 200 * eps)
