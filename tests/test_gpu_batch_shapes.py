"""The batch's shared solve launches over the meshes where their layout changes: one interior
row, a block with neither tile nor line unit (5 rows, at most 9 columns), lines of one unknown
more than a chunk length's most, tall and wide meshes, more reactors than the GPU has room for at
once (blocks cut below a reactor's units)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

MESHES = [(3, 40), (5, 3), (5, 9), (5, 34), (9, 65), (9, 66), (17, 129), (17, 130), (9, 258), (9, 513), (9, 514),
          (257, 40), (17, 1025)]


def reactor(mesh, prec, seed):
    nz, nr = mesh
    return W.scaled(W.config("c1", nz=nz, nr=nr, R=0.2 * (nr - 1) / 512, L=0.025 * (nz - 1) / 128, precision=prec,
                             mg_tol=1e-11, mg_max_cycles=100, seed=seed), 4000)


# few FP64 reactors of long lines, which take what the GPU has to spare, and many, with a block
# or two each and the widest tiles
LONG = [[(33, 1025)], [(9, 130), (17, 300)], [(129, 200)] * 2, [(65, 514)] * 3, [(9, 700)] * 90, [(257, 257)] * 6]


@pytest.mark.parametrize("meshes", LONG, ids=lambda m: "%dx%d of %d" % (*m[0], len(m)))
def test_batched_solves_of_long_fp64_lines(meshes):
    check([reactor(m, "fp64", 10 + k) for k, m in enumerate(meshes)], "fp64")


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("copies", [1, 4])
def test_batched_solves_of_many_shapes(prec, copies):
    check([reactor(m, prec, 10 + c) for c in range(copies) for m in MESHES], prec)


def check(cfgs, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import pic

    hs = [pic.pic_init(c) for c in cfgs]
    b = pic.pic_batch_init(hs)
    for step in (1, 1):  # the second reads what the first left in the flagged words
        assert b.step(step) == [0] * len(hs)
    for c, h in zip(cfgs, hs):
        alone = pic.pic_init(c)
        assert pic.pic_step(alone, 2) == 0
        f, g = pic.pic_get_fields(h), pic.pic_get_fields(alone)
        # both to the solve's tolerance (1e-11 of the largest right-hand side), within the
        # condition of the residual, as in the shape tests of the solve alone; on the mixed path
        # the second step's charge is that of particles pushed in FP32 by the first step's field
        tol = 1e-8 if prec == "fp64" else 2e-5
        assert np.abs(f["phi"] - g["phi"]).max() <= tol * np.abs(g["phi"]).max(), (c["nz"], c["nr"])
        pic.pic_destroy(alone)
    b.close()
