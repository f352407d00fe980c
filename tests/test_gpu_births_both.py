"""Numbering of the newborns of one pass where both species go through the radix sort in one
launch, by many blocks and (a batch's reactor) by one, pass after pass."""
import numpy as np
import pytest

import workloads as W
from oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("births", [(8193, 8193), (20_011, 30_011), (30_011, 9000)])
def test_newborn_ids_of_two_large_species(births, batched):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import pic

    cfg = W.collisionless(W.config("c1", precision="fp64"))
    cfg["split_every"] = 1
    for sp in cfg["species"]:
        sp["n_init"], sp["capacity"] = 40_000, 100_000
    h, o = pic.pic_init(cfg, load=False), Oracle(cfg)
    b = pic.pic_batch_init([h]) if batched else None
    dr = cfg["R"] / (cfg["nr"] - 1)
    for step, mult in enumerate((97, 3)):
        for s, n in enumerate(births):
            # each particle splits once; ids in no order, over three radix digits, then over two
            p = W.random_particles(cfg, s, n, seed=5 + s + 10 * step, hot=0.1, margin=2e-3)
            p["w"] = np.array([o.w_ref(s, int(j)) for j in np.floor(p["r"] / dr)]) * 1.5
            p["id"] = (p["id"] * np.uint64(mult) + np.uint64(13)).astype(np.uint64)
            pic.pic_set_particles(h, s, p)
            o.set_particles(s, p)
        if batched:
            assert b.step(1) == [0]
        else:
            assert pic.pic_step(h, 1) == 0
        o.step(1)
        for s, n in enumerate(births):
            u, v = pic.pic_get_particles(h, s), o.get_particles(s)
            ku, kv = np.argsort(u["id"]), np.argsort(v["id"])
            assert len(kv) >= 2 * n  # (a few cross into a lighter ring first and split in three)
            assert np.array_equal(u["id"][ku], v["id"][kv])
            for f in ("r", "z", "w"):  # FP64 path, one step from equal particles: the same to rounding
                assert np.allclose(u[f][ku], v[f][kv], rtol=1e-10, atol=1e-16)
        assert list(pic.pic_get_counts(h)["next_id"]) == [o.next_id(0), o.next_id(1)]
    if batched:
        b.close()
