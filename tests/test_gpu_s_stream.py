"""The streamed single-precision S product for every replica group (two, four and eight replicas per block) and the
tensor-core product's reduction: q within 1e-5 of S (G psi - b) with the library's own FP64 S, neutral to 1e-12 e."""
import numpy as np
import pytest

from gpu_util import make_ctx, need_gpu, rel_l2, run_update
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def geo():
    need_gpu()
    el = s.graphene_plates(8, 5, 2, 30.0)                 # 640 sites: one full column block and a part of one
    S = make_ctx(el).setup(el).cpm_get_matrix("S").cpu().numpy()
    return el, S


@pytest.mark.parametrize("s_prec", ["fp32", "bf16x3"])
@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 8, 9, 33])
def test_s_product_replica_groups(geo, m, s_prec):
    el, S = geo
    rng = np.random.default_rng(m)
    b = rng.normal(0.0, 0.5, (m, el.n)) + rng.normal(0.0, 2.0, (m, 1)) * el.xyz[:, 2] / 30.0
    psi = np.array([0.0, 1.0])
    q, qt = run_update(make_ctx(el, s_prec=s_prec, k_prec="fp32").setup(el), psi, b)
    ref = (psi[el.group][None] - b) @ S
    for r in range(m):
        assert rel_l2(q[r], ref[r]) <= 1e-5, r
    assert np.abs(qt).max() <= 1e-12
    assert np.abs(q.sum(1)).max() <= 1e-12


@pytest.mark.parametrize("n,s_prec", [(9, "fp64"), (127, "fp32"), (129, "fp64"), (256, "bf16x3"), (515, "fp32"),
                                      (1030, "fp64"), (8203, "fp32")])
def test_s_product_slices(n, s_prec):
    """The reduction's slices: one block, clusters of two, four and eight, empty last slices, more sites than threads."""
    need_gpu()
    el = s.graphene_plates(*((33, 16, 2) if n > 2048 else (8, 9, 2)), 30.0)
    keep = np.unique(np.linspace(0, el.n - 1, n).astype(int))
    el = s.Electrodes(**{**el.__dict__, "xyz": el.xyz[keep], "eta": el.eta[keep], "group": el.group[keep]})
    assert el.n == n
    S = make_ctx(el).setup(el).cpm_get_matrix("S").cpu().numpy()
    rng = np.random.default_rng(n)
    b = rng.normal(0.0, 0.5, (3, n)) + rng.normal(0.0, 2.0, (3, 1)) * el.xyz[:, 2] / 30.0
    psi = np.array([0.0, 1.0])
    q, qt = run_update(make_ctx(el, s_prec=s_prec, k_prec="fp64" if s_prec == "fp64" else "fp32").setup(el), psi, b)
    ref = (psi[el.group][None] - b) @ S
    for r in range(3):
        assert rel_l2(q[r], ref[r]) <= (1e-10 if s_prec == "fp64" else 1e-5), r
    assert np.abs(qt).max() <= 1e-12
    assert np.abs(q.sum(1)).max() <= 1e-12
