"""The two kernels of the 8 x 4 channel set (one warp on four columns, and a warp per column with extra
warps), and the rule that chooses between them and the segments of their march."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle.channel import ChannelGrid, ChannelOracle, ClbChannelOracle  # noqa: E402
from paper_1708_05944_gb300 import vlb  # noqa: E402
from paper_1708_05944_gb300.inputs import perturbation  # noqa: E402
from tests.helpers import rel_err  # noqa: E402

SMALL, HALF = "HH(3;4)xH(3;4)", "HH(3;4)xHH(1;2)"
PRECS = [vlb.VLB_FP64, vlb.VLB_FP32_BULK]


def context(spec, prec, nl, nx, kind):
    c = vlb.Channel(spec, prec, nl, nx, 0.05)
    if kind == "cartesian":
        c.set_formulation(vlb.VLB_CARTESIAN)
    if kind == "flow":
        c.set_flow_rate(0.1)
    return c


# 150 strips of 16 rows: cut into segments they fill the SMs with one-warp CTAs, as one segment each they
# leave them to the kernel with a warp per column
@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("spec,kind", [(SMALL, "vielbein"), (SMALL, "cartesian"), (SMALL, "flow"), (HALF, "vielbein")])
def test_both_kernels_give_the_same_bits(prec, spec, kind):
    out = []
    for variant in (0, 3):  # rows per segment by the host, and one segment
        c = context(spec, prec, 16, 600, kind)
        c.init_equilibrium(1.2, 0.0, 0.05, 1.0)
        F = c.read_f()
        c.set_f((F * perturbation(F.shape, seed=81, amplitude=0.02)).astype(F.dtype))
        c.set_variant(variant)
        c.step(1e-4, 2)
        out.append((c.read_f(), c.wall_density()))
        c.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])


# few strips: the kernel with a warp per column, inlet and outlet in one CTA, in neighbours, and apart; segments
# of three rows and more
@pytest.mark.parametrize("prec,dtype,tol", [(vlb.VLB_FP64, np.float64, 1e-12), (vlb.VLB_FP32_BULK, np.float32, 1e-6)])
@pytest.mark.parametrize("cartesian", [False, True])
@pytest.mark.parametrize("nl,nx", [(3, 4), (5, 8), (11, 20)])
def test_warp_per_column_matches_the_oracle(prec, dtype, tol, cartesian, nl, nx):
    o = (ClbChannelOracle if cartesian else ChannelOracle)(SMALL, ChannelGrid(nl, nx), 0.05, n_in=2.0, n_out=1.0)
    F = o.initial_state()
    F = F * perturbation(F.shape, seed=82, amplitude=0.02)
    c = context(SMALL, prec, nl, nx, "cartesian" if cartesian else "vielbein")
    c.set_f(np.ascontiguousarray(F.transpose(2, 1, 0, 3, 4).reshape(nx * nl, 2, *F.shape[3:])).astype(dtype))
    c.stage(1e-3, 1)
    got = c.read_f().astype(np.float64).reshape(nx, nl, 2, *F.shape[3:]).transpose(2, 1, 0, 3, 4)
    assert rel_err(got, o.stage(1, 1e-3, F, F)) < tol
    c.close()


# 128 strips of 64 rows: a SM holds more than one CTA of the set in either precision, so the march is cut into
# segments until there is more than a CTA per SM
@pytest.mark.parametrize("prec", PRECS)
def test_segments_fill_the_resident_ctas(prec):
    c = vlb.Channel(SMALL, prec, 64, 512, 0.05)
    rows = c.variants()[0][0] // 4
    c.close()
    assert 128 * -(-64 // rows) > torch.cuda.get_device_properties(0).multi_processor_count
