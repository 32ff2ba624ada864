"""vlb_step_static_scratch refuses an output buffer that the stage's bulk copies cannot start at, and takes an
input at any address of its type."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1708_05944_gb300 import vlb  # noqa: E402


@pytest.mark.parametrize("prec,dtype", [(vlb.VLB_FP64, torch.float64), (vlb.VLB_FP32_BULK, torch.float32)])
def test_alignment(prec, dtype):
    c = vlb.Couette("HH(3;4)xH(3;4)", prec, [dict(n_cells=8)], [(0.1, 1.0)], [(0.0, 1.0)], [0.1], [1])
    c.init_equilibrium(1.0, 0.0, 0.0, 1.0)
    f = torch.empty(c.f_shape(), dtype=dtype, device="cuda")
    c.read_f(f)
    n = f.numel()
    a, b = (torch.zeros(n + 1, dtype=dtype, device="cuda") for _ in range(2))
    with pytest.raises(vlb.VlbError) as e:
        c.step_static_scratch(f, b[1:].view(f.shape), 1e-4, 1)
    assert e.value.status == vlb.VLB_ERR_INVALID
    a[1:].copy_(f.flatten())
    c.step_static_scratch(a[1:].view(f.shape), b[:n].view(f.shape), 1e-4, 1)
    out = torch.empty_like(f)
    c.step_static_scratch(f, out, 1e-4, 1)
    torch.cuda.synchronize()
    assert torch.equal(out.flatten(), b[:n])
    c.close()
