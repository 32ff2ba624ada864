"""Fields that are uniform to the last bit over most of the domain, where two of the three WENO-5
indicators vanish at many faces: the result, and that a step takes no longer than on a rough field."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle.channel import ChannelGrid, ChannelOracle, ClbChannelOracle  # noqa: E402
from oracle.couette import CouetteGrid, CouetteOracle, Wall  # noqa: E402
from paper_1708_05944_gb300 import vlb  # noqa: E402
from paper_1708_05944_gb300.inputs import perturbation  # noqa: E402
from tests.helpers import rel_err, to_lib, to_oracle  # noqa: E402

MODEL, SMALL = "HH(4;8)xH(4;12)", "HH(3;4)xH(3;4)"


# Tolerances: a stage's roundings (see test_gpu_kernel_edges.py): 1e-12 in double, 1e-6 in single precision.
@pytest.mark.parametrize("prec,dtype,tol", [(vlb.VLB_FP64, np.float64, 1e-12), (vlb.VLB_FP32_BULK, np.float32, 1e-6)])
@pytest.mark.parametrize("jump", [0.3, 1e-4, 1e-9])
def test_couette_step_profile(prec, dtype, tol, jump):
    n = 24
    o = CouetteOracle(SMALL, CouetteGrid(n, 1.0, 2.0), Wall(0.1), Wall(0.0), 0.1, 1)
    F = o.initial_equilibrium()
    F[:, 9:] *= 1.0 + jump  # one jump between uniform stretches
    F[:, 17] *= 1.0 - jump  # and one cell
    F = F.astype(dtype).astype(np.float64)
    c = vlb.Couette(SMALL, prec, [dict(n_cells=n, r_in=1.0, r_out=2.0)], [(0.1, 1.0)], [(0.0, 1.0)], [0.1], [1])
    c.set_f(to_lib(F).astype(dtype))
    c.stage(1e-3, 1)
    assert rel_err(to_oracle(c.read_f()), o.stage(1, 1e-3, F, F)) < tol
    c.close()


@pytest.mark.parametrize("prec,dtype,tol", [(vlb.VLB_FP64, np.float64, 1e-12), (vlb.VLB_FP32_BULK, np.float32, 1e-6)])
@pytest.mark.parametrize("spec", [SMALL, MODEL])
@pytest.mark.parametrize("cartesian", [False, True])
def test_channel_step_profile(prec, dtype, tol, spec, cartesian):
    nl, nx = 12, 24
    o = (ClbChannelOracle if cartesian else ChannelOracle)(spec, ChannelGrid(nl, nx), 0.05, n_in=2.0, n_out=1.0)
    F = o.initial_state()
    F[:, :, 10:] *= 1.2
    F[:, 5, :] *= 0.9
    F = F.astype(dtype).astype(np.float64)
    c = vlb.Channel(spec, prec, nl, nx, 0.05, n_in=2.0, n_out=1.0)
    if cartesian:
        c.set_formulation(vlb.VLB_CARTESIAN)
    c.set_f(np.ascontiguousarray(F.transpose(2, 1, 0, 3, 4).reshape(nx * nl, 2, *F.shape[3:])).astype(dtype))
    c.stage(1e-4, 1)
    got = c.read_f().astype(np.float64).reshape(nx, nl, 2, *F.shape[3:]).transpose(2, 1, 0, 3, 4)
    assert rel_err(got, o.stage(1, 1e-4, F, F)) < tol
    c.close()


# From rest the interior stays uniform to rounding.  With faces redone a warp at a time a step took
# 1.5 to 2 times that of a rough field; the bound leaves a quarter for the clocks.
@pytest.mark.parametrize("spec,prec,nl,nx", [(MODEL, vlb.VLB_FP32_BULK, 128, 256), (MODEL, vlb.VLB_FP64, 32, 128),
                                             (SMALL, vlb.VLB_FP32_BULK, 256, 512)])
def test_a_step_from_rest_takes_no_longer(spec, prec, nl, nx):
    s = torch.cuda.Stream()
    c = vlb.Channel(spec, prec, nl, nx, 0.05, stream=s.cuda_stream)
    c.init_equilibrium(1.0, 0.0, 0.0, 1.0)
    rough = c.read_f()
    rough = (rough * perturbation(rough.shape, seed=51, amplitude=1e-3)).astype(rough.dtype)

    def ms():
        c.step(2e-5, 6)
        best = np.inf
        for _ in range(3):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record(s)
            c.step(2e-5, 10)
            b.record(s)
            s.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    c.set_f(rough)
    t_rough = ms()
    c.init_equilibrium(1.0, 0.0, 0.0, 1.0)
    t_rest = ms()
    c.close()
    assert t_rest < 1.25 * t_rough
