"""A births buffer far smaller than the mesh: the launch that numbers the newborns and clears the
pass's accumulators takes its blocks from the mesh, and gives the steps of a large buffer."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh", [(33, 65), (65, 64), (65, 66), (129, 513)])  # 1 and 2 blocks' nodes, many
def test_small_births_capacity(mesh):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import pic

    nz, nr = mesh
    cfg = W.scaled(W.config("c1", nz=nz, nr=nr, R=0.05 * (nr - 1) / 64, precision="fp64", split_every=0), 40_000)
    cfg["gas"] = dict(cfg["gas"], p_Pa=40.0)
    small, large = pic.pic_init(dict(cfg, births_capacity=300)), pic.pic_init(cfg)
    for h in (small, large):
        assert pic.pic_step(h, 5) == 0
    a, b = pic.pic_get_deposit(small), pic.pic_get_deposit(large)
    for x, y in ((a[k], b[k]) for k in ("Ne", "Ni")):  # FP64 sums of the same weights in another order
        assert np.abs(x - y).max() <= 1e-10 * np.abs(y).max()
    ca, cb = pic.pic_get_counts(small), pic.pic_get_counts(large)
    assert list(ca["n_alive"]) == list(cb["n_alive"]) and list(ca["next_id"]) == list(cb["next_id"])
