"""A call that fails for capacity, and what the handle does next: it is at the last completed
step, takes that step again, and goes on as a handle that was stepped that far and no further."""
import numpy as np
import pytest

import workloads as W
from oracle import Oracle

pytestmark = pytest.mark.gpu

FIELDS = ("r", "z", "vr", "vt", "vz", "w")
SHORT = {"capacity": 35_000, "births": 9_000}


def by_id(p):
    o = np.argsort(p["id"], kind="stable")
    return {k: np.asarray(v)[o] for k, v in p.items()}


def nerr(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def pair(short, split_every=3):
    """Two handles of one reactor: electrons ionise in every step (1200 newborns) and split in every
    third (46,000, to 68,000 electrons), which the first handle cannot hold."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import pic

    cfg = W.config("c1", precision="fp64", split_every=split_every)
    cfg["gas"] = dict(cfg["gas"], p_Pa=100.0)
    for sp in cfg["species"]:
        sp["n_init"], sp["capacity"], sp["n0"] = 0, 400_000, 1e12  # (a weak plasma: no sheath field)
    o = Oracle(cfg, capacity=64)
    dr = cfg["R"] / (cfg["nr"] - 1)
    parts = [W.random_particles(cfg, s, 20_000 if s == 0 else 1000, seed=61 + s, hot=4.0 if s == 0 else 1.0,
                                margin=3e-3) for s in (0, 1)]
    for s, p in enumerate(parts):
        w = np.array([o.w_ref(s, j) for j in range(cfg["nr"] - 1)])
        p["w"] = w[np.floor(p["r"] / dr).astype(int)] * (2.5 if s == 0 else 0.5)
    small = dict(cfg, species=[dict(sp) for sp in cfg["species"]])
    if short == "births":
        small["births_capacity"] = SHORT[short]
    else:
        small["species"][0]["capacity"] = SHORT[short]
    hs = [pic.pic_init(c, load=False) for c in (small, cfg)]
    for h in hs:
        for s, p in enumerate(parts):
            pic.pic_set_particles(h, s, p)
    return pic, hs[0], hs[1]


def same(pic, a, b, grids=("rho", "chi")):
    ca, cb = pic.pic_get_counts(a), pic.pic_get_counts(b)
    assert ca["step"] == cb["step"] and list(ca["n_alive"]) == list(cb["n_alive"])
    assert list(ca["next_id"]) == list(cb["next_id"])
    for s in (0, 1):
        u, v = by_id(pic.pic_get_particles(a, s)), by_id(pic.pic_get_particles(b, s))
        assert np.array_equal(u["id"], v["id"]), s
        for k in FIELDS:  # the same FP64 arithmetic, but for the solves' starting values (tolerance 1e-10)
            assert nerr(u[k], v[k]) < 1e-8, (s, k)
    fa, fb = pic.pic_get_fields(a), pic.pic_get_fields(b)
    for k in grids:
        assert nerr(fa[k], fb[k]) < 1e-8, k


@pytest.mark.parametrize("short", ["capacity", "births"])
def test_a_failed_step_fails_again_and_leaves_the_step_number(short):
    pic, h, ref = pair(short)
    assert pic.pic_step(h, 2) == 0 and pic.pic_step(ref, 2) == 0
    for n in (1, 1, 1):  # the third step splits
        with pytest.raises(pic.PicError) as err:
            pic.pic_step(h, n)
        assert err.value.status == pic.PIC_ERR_CAPACITY
        same(pic, h, ref)


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("short", ["capacity", "births"])
def test_a_failed_call_of_several_steps_keeps_births_and_deposit(short, batched):
    """The pass that overflows is followed by further steps of its call, whose kernels find out."""
    pic, h, ref = pair(short)
    assert pic.pic_step(ref, 2) == 0
    b = pic.pic_batch_init([h]) if batched else None
    for _ in range(2):
        if batched:
            with pytest.raises(pic.PicError):
                b.step(5)
        else:
            with pytest.raises(pic.PicError) as err:
                pic.pic_step(h, 5)
            assert err.value.status == pic.PIC_ERR_CAPACITY
        same(pic, h, ref)
    for x in (h, ref):  # on from there, from a step that does not split
        pic.pic_set_step(x, 0)
        assert pic.pic_step(x, 2) == 0
    same(pic, h, ref, grids=("rho", "chi", "phi"))
    if batched:
        b.close()
