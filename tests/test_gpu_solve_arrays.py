"""The stand-alone solve's device arrays: what it can read where it lies and what it copies first
give the same potential, also where the output takes an input's place."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("where", ["device", "odd offset", "pinned host", "output over rho"])
def test_device_arrays(prec, where):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import pic

    cfg = W.scaled(W.config("c1", precision=prec), 0)
    chi = W.random_grid(cfg, seed=1, scale=2.0)
    rho = 1e-5 * (W.random_grid(cfg, seed=2, smooth=False) - 0.5)
    h = pic.pic_init(cfg, load=False)
    ref = pic.pic_field_solve(h, rho, chi, 60.0)

    def put(x):
        if where == "pinned host":
            return torch.from_numpy(x.copy()).pin_memory()
        n = 1 if where == "odd offset" else 0  # 8 bytes past the allocation's start
        t = torch.zeros(x.size + n, dtype=torch.float64, device="cuda")
        t[n:] = torch.from_numpy(x).flatten().cuda()
        return t[n:]

    r, c = put(rho), put(chi)
    phi = r if where == "output over rho" else torch.zeros(cfg["nz"], cfg["nr"], dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    out = pic.pic_field_solve_device(h, r.data_ptr(), c.data_ptr(), 60.0, phi.data_ptr())
    torch.cuda.synchronize()
    assert out[-1] == ref[3] == 0
    assert np.array_equal(phi.cpu().numpy().reshape(ref[0].shape), ref[0])
