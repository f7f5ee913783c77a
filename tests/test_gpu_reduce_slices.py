"""The reduction behind the streamed and the tensor-core S product, at the edges of its blocks per replica (sixteen, eight,
four, two, one), with slices beyond one pass of a block's threads, and with the splits added beforehand: q within 1e-5
of S (G psi - b) with the library's own FP64 S (1e-10 in FP64), neutral to 1e-12 e."""
import numpy as np
import pytest

from gpu_util import dev, make_ctx, need_gpu, torch
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def geo():
    need_gpu()
    held = {}

    def get(n):
        if n not in held:
            el = s.graphene_plates(*((33, 20, 2) if n > 2048 else (16, 9, 2)), 30.0)
            keep = np.unique(np.linspace(0, el.n - 1, n).astype(int))
            el = s.Electrodes(**{**el.__dict__, "xyz": el.xyz[keep], "eta": el.eta[keep], "group": el.group[keep]})
            assert el.n == n
            ctx = make_ctx(el, k_prec="fp32").setup(el)
            held.clear()
            held[n] = (el, ctx, ctx.cpm_get_matrix("S"))
        return held[n]
    return get


@pytest.mark.parametrize("n,m,s_prec", [
    (1029, 4, "fp32"), (1029, 5, "fp64"), (1029, 38, "fp32"), (1029, 39, "bf16x3"), (1029, 76, "fp64"), (1029, 77, "fp32"),
    (1029, 152, "bf16x3"), (1029, 153, "fp32"), (1029, 305, "bf16x3"), (1029, 305, "fp64"),
    (2049, 153, "fp32"), (2049, 20, "bf16x3"),
    (10241, 1, "fp32"), (10241, 7, "bf16x3"), (10244, 5, "fp32"), (10244, 19, "fp32"), (10244, 20, "fp32"),
    (10244, 3, "fp64"), (10244, 6, "bf16x3")])
def test_slices(geo, n, m, s_prec):
    el, ctx, S = geo(n)
    ctx.cpm_set_s_prec(s_prec)
    rng = np.random.default_rng(n + m)
    b = dev(rng.normal(0.0, 0.5, (m, n)) + rng.normal(0.0, 2.0, (m, 1)) * el.xyz[:, 2] / 30.0)
    psi = dev(rng.normal(0.0, 1.0, (m, 2)))
    q = torch.empty((m, n), dtype=torch.float64, device="cuda")
    qt = torch.empty((m,), dtype=torch.float64, device="cuda")
    ctx.cpm_update(m, psi, b, q, qt)
    ref = (psi[:, torch.as_tensor(el.group, dtype=torch.long, device="cuda")] - b) @ S
    err = (q - ref).norm(dim=1) / ref.norm(dim=1)
    assert float(err.max()) <= (1e-10 if s_prec == "fp64" else 1e-5)
    assert float(qt.abs().max()) <= 1e-12
    assert float(q.sum(1).abs().max()) <= 1e-12
