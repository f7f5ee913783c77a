"""The FP64 S product for the row splits of small, odd and large electrodes and every replica group (one, two, four and eight
replicas per block): q within 1e-12 of S (G psi - b) with the library's own S."""
import numpy as np
import pytest

from gpu_util import make_ctx, need_gpu, rel_l2, run_update
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 16, 17, 257, 640, 2050])
def test_fp64_product(n):
    need_gpu()
    el = s.graphene_plates(*((16, 9, 2) if n > 640 else (8, 5, 2)), 30.0)
    keep = np.unique(np.linspace(0, el.n - 1, n).astype(int))
    el = s.Electrodes(**{**el.__dict__, "xyz": el.xyz[keep], "eta": el.eta[keep], "group": el.group[keep]})
    ctx = make_ctx(el).setup(el)
    S = ctx.cpm_get_matrix("S").cpu().numpy()
    psi = np.array([0.0, 1.0])
    for m in (1, 2, 3, 4, 5, 8, 9, 64):
        rng = np.random.default_rng(100 * n + m)
        b = rng.normal(0.0, 1.0, (m, n))
        q, qt = run_update(ctx, psi, b)
        ref = (psi[el.group][None] - b) @ S
        if n == 1:   # S = 0: the charge-neutral projection leaves one site without a charge
            assert np.abs(q).max() <= 1e-12
        else:
            assert rel_l2(q, ref) <= 1e-12, m
        assert np.abs(qt).max() <= 1e-12
