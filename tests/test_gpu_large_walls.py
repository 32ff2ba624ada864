"""Wall densities of the large-set stage, which the cell next to a wall computes for the update: ragged
instances, both walls, and more cells than CTAs of the cell kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1708_05944_gb300 import vlb  # noqa: E402
from tests.helpers import make_case, rel_err, to_lib, to_oracle  # noqa: E402


# 1e-12 of the largest value after a stage in double precision, as in test_gpu_kernel_edges.py; single
# precision: 1e-6 of the largest population there, and n_w is a sum of fluxes of such populations
@pytest.mark.parametrize("prec,dtype,tol", [(vlb.VLB_FP64, np.float64, 1e-12), (vlb.VLB_FP32_BULK, np.float32, 1e-6)])
@pytest.mark.parametrize("spec,sizes", [("HH(3;17)xHH(1;2)", (3, 5, 4)), ("HH(3;17)xHH(1;2)", (700, 640)),
                                        ("HH(3;20)xH(3;6)", (3, 17))])
def test_wall_densities(prec, dtype, tol, spec, sizes):
    cases = [make_case(spec, n, u_in=0.1 * (k + 1), u_out=-0.05 * k, T_out=1.0 + 0.02 * k, kn=0.1, seed=71 + k)
             for k, n in enumerate(sizes)]
    c = vlb.Couette(spec, prec, [g for _, _, g in cases], [(0.1 * (k + 1), 1.0) for k in range(len(sizes))],
                    [(-0.05 * k, 1.0 + 0.02 * k) for k in range(len(sizes))], [0.1] * len(sizes), [1] * len(sizes))
    c.set_f(np.concatenate([to_lib(F) for _, F, _ in cases]).astype(dtype))
    c.stage(1e-5, 1)
    got, nw, at = c.read_f(), c.wall_density(), 0
    c.close()
    for k, (o, F, _) in enumerate(cases):
        ref = o.stage(1, 1e-5, F, F)
        assert rel_err(to_oracle(got[at:at + sizes[k]]), ref) < tol
        assert np.abs(nw[k] - np.asarray(o.last_nw)).max() < tol
        at += sizes[k]
