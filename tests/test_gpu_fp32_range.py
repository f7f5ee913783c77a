"""Sums of single-precision partials that leave FP32's range while every partial is inside it: b of the single-precision
paths and q of the tensor-core product stay finite and agree with FP64 (2e-6 and 1e-5)."""
import numpy as np
import pytest

from gpu_util import dev, make_ctx, need_gpu, rel_l2, run_bvec, run_update, torch
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu
FMAX = float(np.finfo(np.float32).max)


@pytest.mark.parametrize("k_prec", ["fp32", "f16x2"])
@pytest.mark.parametrize("shared", [True, False])
def test_b(k_prec, shared):
    need_gpu()
    # a narrow splitting: the reciprocal part at the charge's own place is 2 alpha / sqrt(pi) = 1.7 Q
    el = s.au111_slab(seed_layers=2, nx=6, ny=6, gap=12.0, alpha=1.5, rcut=4.0)
    el = s.Electrodes(**{**el.__dict__, "eta": np.full(el.n, 1.9)})
    if not shared:
        xyz = el.xyz.copy()
        xyz[:, 2] += 0.01 * np.arange(el.n) / el.n
        el = s.Electrodes(**{**el.__dict__, "xyz": xyz})
    e = s.Electrolyte(xyz=el.xyz[40:41] + 0.02, Q=np.array([2.4e38]))
    b = []
    for kp in ("fp64", k_prec):
        ctx = make_ctx(el, k_prec=kp)
        ctx.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
        b.append(run_bvec(ctx, [e, s.Electrolyte(xyz=e.xyz, Q=e.Q / 2.0 ** 100)]))
    assert b[0][0, 40] / 14.399645 > FMAX
    assert np.isfinite(b[1]).all()
    for r in range(2):
        assert rel_l2(b[1][r] / 2.0 ** 100, b[0][r] / 2.0 ** 100) <= 2e-6, r


def test_q():
    """Four splits of one layer of 256 sites each, every one with 0.9 of FP32's largest value for every q_i: S = p p^T / 256
    (imported), b = 0.9 p, p = +-1 without a mean in any layer."""
    need_gpu()
    el = s.graphene_plates(8, 8, 2, 30.0)
    ctx = make_ctx(el, k_prec="fp32").setup(el)
    n, m, splits = el.n, 8, 4
    layers = np.unique(el.xyz[:, 2], return_inverse=True)[1].reshape(splits, 256)
    assert (layers == layers[:, :1]).all() and len(np.unique(layers[:, 0])) == splits
    p = np.random.default_rng(4).permuted(np.tile(np.repeat([1.0, -1.0], 128), (splits, 1)), axis=1).ravel()
    buf = ctx.cpm_export().numpy()
    held = buf[72:72 + 8 * n * (n + el.n_groups)].view(np.float64)
    held[:n * n] = np.outer(p, p).ravel() / 256.0
    held[n * n:] = 0.0
    ctx.cpm_import(buf)
    ctx.cpm_set_s_prec("bf16x3")
    ctx.cpm_gemm_set_plan(m, 32, 2, splits)
    f = np.array([0.9, 1e-3, -0.9, 0.2, 0.5, -0.5, 1e-30, 0.0])
    q, qt = run_update(ctx, np.zeros(2), f[:, None] * FMAX * p)
    assert np.isfinite(q).all()
    assert np.abs(q / FMAX + 4.0 * f[:, None] * p).max() <= 1e-5
    assert np.abs(qt / FMAX).max() <= 1e-9
