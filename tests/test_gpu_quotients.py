"""FP64 quotients by an inverse and a residual correction: those of a division, in the particle
pass's own functions over the divisors it has, and on the grids."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "pmath.cuh"
using namespace pic;
__global__ void k(const double *a, const double *b, double *q, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) q[i] = m_quot(a[i], b[i], m_inv(b[i]));
}
__global__ void ks(const int *j, const double *o, const double *inv_t, double *s, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    shape_r<double>(PIC_WEIGHT_ZR2, j[i], o[i], s[4 * i], s[4 * i + 1], inv_t);
    shape_r<double>(PIC_WEIGHT_ZR2, j[i], o[i], s[4 * i + 2], s[4 * i + 3]);
}
extern "C" int quotients(const double *a, const double *b, double *q, int n) {
    k<<<(n + 255) / 256, 256>>>(a, b, q, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int shapes(const int *j, const double *o, const double *inv_t, double *s, int n) {
    ks<<<(n + 255) / 256, 256>>>(j, o, inv_t, s, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def env(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import build as B
    from paper_1001_2969_gb300.build import ARCH, CSRC, INCLUDE, _nvcc

    B()
    if not (os.path.exists(_nvcc()) or shutil.which(_nvcc())):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("quot")
    (d / "quot.cu").write_text(SOURCE)
    subprocess.check_call([_nvcc(), *ARCH, "-O3", "-std=c++17", "-I", INCLUDE, "-I", CSRC, "-shared", "-Xcompiler",
                           "-fPIC", "-o", str(d / "quot.so"), str(d / "quot.cu")])
    return torch, C.CDLL(str(d / "quot.so"))


def ptr(t):
    return C.c_void_p(t.data_ptr())


def same_as_division(q, a, b):
    """At most one unit in the last place, and that for no more than one in a million (a tie's
    neighbourhood is 2^-51 units wide; an uncorrected product is off for one in four)."""
    ref = a / b
    assert np.all(np.abs(q - ref) <= np.spacing(np.abs(ref)))
    assert np.count_nonzero(q != ref) <= 1e-6 * q.size + 1


@pytest.mark.parametrize("divisor", ["root", "odd"])
def test_quotients_are_those_of_a_division(env, divisor):
    torch, lib = env
    n, rng = 1_000_000, np.random.default_rng(7)
    b = np.sqrt(10.0 ** rng.uniform(-18, 18, n)) if divisor == "root" else 2.0 * rng.integers(0, 1025, n) + 1.0
    a = rng.normal(size=n) * 10.0 ** rng.uniform(-12, 12, n)
    a[:5] = (0.0, -0.0, b[2], -b[3], 3.0 * b[4])
    ta, tb, q = torch.tensor(a, device="cuda"), torch.tensor(b, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.quotients(ptr(ta), ptr(tb), ptr(q), n) == 0
    same_as_division(q.cpu().numpy(), a, b)


def test_radial_shapes_with_and_without_the_table(env):
    torch, lib = env
    n, rng = 1_000_000, np.random.default_rng(8)
    j = rng.integers(0, 1024, n).astype(np.int32)
    o = rng.uniform(0.0, 1.0, n)
    j[:3], o[:3] = (0, 0, 1023), (0.0, np.nextafter(1.0, 0.0), 0.0)
    tj, to = torch.tensor(j, device="cuda"), torch.tensor(o, device="cuda")
    inv = 1.0 / (2.0 * torch.arange(1024, dtype=torch.float64) + 1.0)
    ti, s = inv.cuda(), torch.zeros(n, 4, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.shapes(ptr(tj), ptr(to), ptr(ti), ptr(s), n) == 0
    s = s.cpu().numpy()
    assert np.array_equal(s[:, :2], s[:, 2:])
    t = 2.0 * j + 1.0
    same_as_division(s[:, 1], o * (t - 1.0 + o), t)
    same_as_division(s[:, 0], (1.0 - o) * (t + o), t)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_field_is_the_divided_difference(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1001_2969_gb300 import pic

    cfg = W.scaled(W.config("c1", precision=prec, nr=130, R=0.0501, L=0.0203), 20_000)
    h = pic.pic_init(cfg)
    pic.pic_set_step(h, 77)
    pic.pic_step(h, 1)
    f = pic.pic_get_fields(h)
    phi, dz, dr = f["phi"], cfg["L"] / (cfg["nz"] - 1), cfg["R"] / (cfg["nr"] - 1)
    Ez = np.concatenate([(phi[:1] - phi[1:2]) / dz, (phi[:-2] - phi[2:]) / (2 * dz), (phi[-2:-1] - phi[-1:]) / dz])
    Er = np.concatenate([0 * phi[:, :1], (phi[:, :-2] - phi[:, 2:]) / (2 * dr), (phi[:, -2:-1] - phi[:, -1:]) / dr], 1)
    for a, b in ((f["Ez"], Ez), (f["Er"], Er)):
        assert np.all(np.abs(a - b) <= np.spacing(np.abs(b)))
        assert np.count_nonzero(a != b) <= 1
