"""The one-launch solve at the sizes where its layout changes: lines of one unknown more than a
chunk length's most (32 M, in FP64 128 M'), the fewest and the most unknowns, more residual
tiles than SMs (wider tiles), more line units than blocks (factor slots reloaded), tall meshes
(narrower tiles)."""
import numpy as np
import pytest

import workloads as W
from oracle import Oracle

pytestmark = pytest.mark.gpu

MESHES = [(5, 3), (5, 34), (9, 65), (9, 66), (17, 129), (17, 130), (33, 257), (33, 258), (9, 513), (9, 514),
          (17, 701), (5, 1025), (513, 40), (1025, 20)]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("mesh", MESHES)
def test_solve_shapes(mesh, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import pic

    nz, nr = mesh
    # FP64: three cycles of the oracle's own iteration, the same to rounding (eps times the few
    # hundred operations of a line, times cycles); mixed: both converged, each to within the
    # condition of its residual, as in the parity test of the solve
    fixed = prec == "fp64"
    cfg = W.scaled(W.config("c1", nz=nz, nr=nr, R=0.2 * (nr - 1) / 512, L=0.025 * (nz - 1) / 128, precision=prec,
                            mg_tol=0.0 if fixed else 1e-11, mg_max_cycles=3 if fixed else 100), 0)
    h, o = pic.pic_init(cfg, load=False), Oracle(cfg)
    chi = W.random_grid(cfg, seed=nz, scale=2.0)
    rho = 1e-5 * (W.random_grid(cfg, seed=nr, smooth=False) - 0.5)
    phi, cyc, res, st = pic.pic_field_solve(h, rho, chi, 80.0)
    again = pic.pic_field_solve(h, rho, chi, 80.0)[0]  # the flagged words of the solve before are not taken
    o.set_grid("chi", chi)
    o.set_grid("rho", rho)
    o.set_grid("phi", np.zeros((nz, nr)))
    ost, ocyc, _ = o.solve(80.0, tol=0.0 if fixed else 1e-13, max_cycles=3 if fixed else 200)
    assert st == 0 and ost == 0
    ref = o.grid("phi")
    assert np.abs(phi - ref).max() <= (1e-11 if fixed else 1e-8) * np.abs(ref).max()
    assert np.array_equal(phi, again)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_solve_after_a_solve_that_was_not_finite(prec):
    """What a solve of non-finite charge leaves in the handle's workspace does not reach the next."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import pic

    cfg = W.scaled(W.config("c1", precision=prec, mg_max_cycles=30), 0)
    chi = W.random_grid(cfg, seed=1, scale=2.0)
    rho = 1e-5 * (W.random_grid(cfg, seed=2, smooth=False) - 0.5)
    bad = rho.copy()
    bad[7, 11] = np.nan
    fresh = pic.pic_field_solve(pic.pic_init(cfg, load=False), rho, chi, 60.0)
    h = pic.pic_init(cfg, load=False)
    assert pic.pic_field_solve(h, bad, chi, 60.0)[3] == pic.PIC_ERR_NOT_CONVERGED
    phi, cyc, _, st = pic.pic_field_solve(h, rho, chi, 60.0)
    assert st == fresh[3] == 0 and cyc == fresh[1] and np.array_equal(phi, fresh[0])
