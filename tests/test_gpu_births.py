"""Numbering of the newborns of one pass (parent id, birth slot order) at the sizes where its
kernels change: one birth, a block's keys and one more, a shared-memory tile of keys and one
more, the most the counting kernel takes and one more (the radix sort), both species apart."""
import numpy as np
import pytest

import workloads as W
from oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("births", [(1, 0), (16, 17), (2048, 2049), (8192, 8193), (20_011, 8192)])
def test_newborn_ids(births):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import pic

    cfg = W.collisionless(W.config("c1", precision="fp64"))
    cfg["split_every"] = 1
    for sp in cfg["species"]:
        sp["n_init"], sp["capacity"] = 40_000, 100_000
    h, o = pic.pic_init(cfg, load=False), Oracle(cfg)
    dr = cfg["R"] / (cfg["nr"] - 1)
    for s, n in enumerate(births):
        # each particle splits once; the ids are spread over three radix digits, in no order
        p = W.random_particles(cfg, s, n, seed=5 + s, hot=0.1, margin=2e-3)
        p["w"] = np.array([o.w_ref(s, int(j)) for j in np.floor(p["r"] / dr)]) * 1.5
        p["id"] = (p["id"] * np.uint64(97) + np.uint64(13)).astype(np.uint64)
        pic.pic_set_particles(h, s, p)
        o.set_particles(s, p)
    pic.pic_step(h, 1)
    o.step(1)
    for s, n in enumerate(births):
        a, b = pic.pic_get_particles(h, s), o.get_particles(s)
        ka, kb = np.argsort(a["id"]), np.argsort(b["id"])
        assert len(ka) == 2 * n
        assert np.array_equal(a["id"][ka], b["id"][kb])
        for f in ("r", "z", "w"):  # FP64 path, one step: the same arithmetic to rounding
            assert np.allclose(a[f][ka], b[f][kb], rtol=1e-10, atol=1e-16)
    assert list(pic.pic_get_counts(h)["next_id"]) == [o.next_id(0), o.next_id(1)]
