"""The kernels chosen by velocity set, size, type and alignment, at the edges of what each takes:
the channel march for a half-range wall-parallel axis and on both sides of its extra-warp rule, the
one-cell and remainder tiles of the Couette stage, the Shakhov kernel of the fixed sets, the
large-set launches and the two forms of the layout conversion.

Tolerances.  Double precision: 1e-12 of the largest value after a stage (some 1e3 operations of
2^-53 in a force row, against 1).  Single precision: a stage rounds the stored deviation (2^-24 of
a population) and adds dt L, whose terms carry some ten roundings of 2^-24 of dt (1 / tau + p / ds +
|K| / r) <= 0.2 times a population here; 1e-6 of the largest population is five times the sum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle.channel import ChannelGrid, ChannelOracle  # noqa: E402
from oracle.couette import CouetteGrid, CouetteOracle, Wall  # noqa: E402
from paper_1708_05944_gb300 import vlb  # noqa: E402
from paper_1708_05944_gb300.inputs import perturbation  # noqa: E402
from tests.helpers import make_case, rel_err, to_lib, to_oracle  # noqa: E402

PRECS = [vlb.VLB_FP64, vlb.VLB_FP32_BULK]


def dtype_tol(prec):
    return (np.float64, 1e-12) if prec == vlb.VLB_FP64 else (np.float32, 1e-6)


# 8 x 4 velocities: 1217 strips are beyond the grids that get extra warps in either precision
@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("spec,nl,nx", [("HH(4;8)xHH(4;6)", 3, 4), ("HH(4;8)xHH(4;6)", 6, 20), ("HH(3;4)xHH(1;2)", 5, 12),
                                        ("HH(3;4)xH(3;4)", 4, 20), ("HH(3;4)xH(3;4)", 3, 4 * 1217)])
def test_channel_stage(prec, spec, nl, nx):
    o = ChannelOracle(spec, ChannelGrid(nl, nx), 0.05, n_in=2.0, n_out=1.0)
    F = o.initial_state()
    F = F * perturbation(F.shape, seed=41, amplitude=0.02)
    dtype, tol = dtype_tol(prec)
    c = vlb.Channel(spec, prec, nl, nx, 0.05, n_in=2.0, n_out=1.0)
    c.set_f(np.ascontiguousarray(F.transpose(2, 1, 0, 3, 4).reshape(nx * nl, *F.shape[0:1], *F.shape[3:])).astype(dtype))
    c.stage(1e-3, 1)
    got = c.read_f().astype(np.float64).reshape(nx, nl, 2, *F.shape[3:]).transpose(2, 1, 0, 3, 4)
    assert rel_err(got, o.stage(1, 1e-3, F, F)) < tol
    c.close()


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("spec", ["HH(4;8)xH(4;20)", "HH(4;8)xH(4;12)", "HH(3;4)xH(3;4)", "H(4;5)xH(4;5)"])
@pytest.mark.parametrize("n", [3, 4, 5, 153])
def test_couette_stage(prec, spec, n):
    o, F, grid = make_case(spec, n, u_in=0.2, u_out=-0.05, T_out=1.05, kn=0.1, seed=42)
    dtype, tol = dtype_tol(prec)
    c = vlb.Couette(spec, prec, [grid], [(0.2, 1.0)], [(-0.05, 1.05)], [0.1], [1])
    c.set_f(to_lib(F).astype(dtype))
    c.stage(1e-4, 1)
    assert rel_err(to_oracle(c.read_f()), o.stage(1, 1e-4, F, F)) < tol
    c.close()


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("spec,n", [("HH(4;8)xH(4;12)", 3), ("HH(4;8)xHH(4;10)", 5), ("HH(3;4)xH(3;4)", 3),
                                    ("HH(3;4)xH(3;5)", 4)])
def test_shakhov_stage(prec, spec, n):
    o = CouetteOracle(spec, CouetteGrid(n, 1.0, 2.0), Wall(0.2, 1.0), Wall(0.0, 1.05), 0.1, 1, prandtl=2.0 / 3.0)
    F = o.initial_equilibrium()
    F = F * perturbation(F.shape, seed=43, amplitude=0.03)
    dtype, tol = dtype_tol(prec)
    c = vlb.Couette(spec, prec, [dict(n_cells=n, r_in=1.0, r_out=2.0)], [(0.2, 1.0)], [(0.0, 1.05)], [0.1], [1])
    c.set_collision(vlb.VLB_SHAKHOV, 2.0 / 3.0)
    c.set_f(to_lib(F).astype(dtype))
    c.stage(1e-4, 1)
    assert rel_err(to_oracle(c.read_f()), o.stage(1, 1e-4, F, F)) < tol
    c.close()


@pytest.mark.parametrize("prec", PRECS)
def test_large_set_stage_of_three_cells(prec):
    spec = "HH(3;17)xHH(2;3)"
    o, F, grid = make_case(spec, 3, u_in=0.2, kn=0.1, seed=44)
    dtype, tol = dtype_tol(prec)
    c = vlb.Couette(spec, prec, [grid], [(0.2, 1.0)], [(0.0, 1.0)], [0.1], [1])
    c.set_f(to_lib(F).astype(dtype))
    c.stage(1e-4, 1)
    assert rel_err(to_oracle(c.read_f()), o.stage(1, 1e-4, F, F)) < tol
    c.close()


# 25 velocities: padded rows; 32 and 320: pairs of velocities where the buffer is aligned to 8 bytes
@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("spec", ["H(4;5)xH(4;5)", "HH(3;4)xH(3;4)", "HH(4;8)xH(4;20)"])
def test_layout_conversion(prec, spec):
    c = vlb.Couette(spec, prec, [dict(n_cells=n, r_in=1.0, r_out=2.0) for n in (3, 14)], [(0.1, 1.0)] * 2,
                    [(0.0, 1.0)] * 2, [0.1] * 2, [1] * 2)
    dtype = torch.float64 if prec == vlb.VLB_FP64 else torch.float32
    g = torch.Generator().manual_seed(45)
    x = torch.rand(c.f_shape(), generator=g, dtype=torch.float64).to(dtype)
    x[0, 0, 0, :3] = torch.tensor([float("inf"), float("-inf"), float("nan")], dtype=dtype)
    x[1, 1, 1, :3] = torch.tensor([0.0, 3e38, -3e38], dtype=dtype)
    n = x.numel()
    back = []
    for off in (0, 1):  # the second at one value past an aligned address
        src, dst = (torch.zeros(n + 1, dtype=dtype, device="cuda") for _ in range(2))
        a, b = src[off:off + n].view(x.shape), dst[off:off + n].view(x.shape)
        a.copy_(x)
        c.set_f(a)
        c.read_f(b)
        torch.cuda.synchronize()
        assert float(dst[n if off == 0 else 0]) == 0.0  # nothing beyond the caller's values
        back.append(b.cpu())
    np.testing.assert_array_equal(back[0].numpy(), back[1].numpy())
    # D = x - R and D + R round once each: 2^-p (|D| + |x|), |D| <= |x| + 1, and 1 % for higher orders
    eps = 2.0 ** (-53 if prec == vlb.VLB_FP64 else -24)
    ok = torch.isfinite(x)
    np.testing.assert_array_equal(back[0][~ok].numpy(), x[~ok].numpy())
    err = (back[0][ok].double() - x[ok].double()).abs()
    assert bool((err <= 1.01 * eps * (2 * x[ok].double().abs() + 1)).all())
    c.close()
