"""A cell sort that fails in the middle of a call, beside the next step's field solve: whatever
the solve was doing then, the handle's next solves are those of a handle that never failed."""
import numpy as np
import pytest

import workloads as W
from oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("circuit", [0.0, 1e-9])
def test_solves_after_a_sort_that_failed_beside_a_solve(prec, circuit):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import pic

    cfg = W.collisionless(W.config("c1", precision=prec, circuit_C=circuit))
    cfg["split_every"] = 1
    for sp in cfg["species"]:
        sp["n_init"], sp["capacity"] = 0, 30_050
    o = Oracle(cfg)
    dr = cfg["R"] / (cfg["nr"] - 1)
    p = [W.random_particles(cfg, s, 30_000 if s == 0 else 1000, seed=41 + s, hot=0.1, margin=2e-3) for s in (0, 1)]
    p[0]["w"] = np.array([o.w_ref(0, int(j)) for j in np.floor(p[0]["r"] / dr)]) * 3.5  # every electron splits
    chi = W.random_grid(cfg, seed=1, scale=2.0)
    rho = 1e-5 * (W.random_grid(cfg, seed=2, smooth=False) - 0.5)
    ref = pic.pic_field_solve(pic.pic_init(cfg, load=False), rho, chi, 60.0)
    assert ref[3] == 0
    h = pic.pic_init(cfg, load=False)
    for s in (0, 1):
        pic.pic_set_particles(h, s, p[s])
    for _ in range(20):
        # the first pass overflows; its sort finds out beside the second step's solve
        with pytest.raises(pic.PicError) as err:
            pic.pic_step(h, 3)
        assert err.value.status == pic.PIC_ERR_CAPACITY
        assert pic.pic_get_counts(h)["step"] == 0
        got = pic.pic_field_solve(h, rho, chi, 60.0)
        assert got[3] == 0 and got[1] == ref[1] and np.array_equal(got[0], ref[0])
