"""The two site stages of b on electrodes whose sites share some heights, on both sides of the line that the number of
heights and of replicas draws between them: every replica within 2e-6 of the FP64 b of the same library, which is
compared with the oracle at sampled sites (1e-11)."""
import numpy as np
import pytest

from gpu_util import dev, make_ctx, need_gpu, rel_l2, run_bvec, torch
from oracle import cpm_oracle as o
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu


def _on_heights(el, heights):
    """The same sites, in the order of z, on so many heights."""
    order = np.argsort(el.xyz[:, 2], kind="stable")
    z = np.empty(el.n)
    for u, part in enumerate(np.array_split(order, heights)):
        z[part] = el.xyz[part[0], 2] + 0.3 * np.sin(1.7 * u + 0.2)
    xyz = el.xyz.copy()
    xyz[:, 2] = z
    assert len(np.unique(z)) == heights
    return s.Electrodes(**{**el.__dict__, "xyz": xyz})


def _ctx(el, k_prec):
    ctx = make_ctx(el, k_prec=k_prec)
    ctx.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
    return ctx


@pytest.mark.parametrize("k_prec,heights,replicas", [
    ("f16x2", 64, (1, 2, 3)), ("f16x2", 128, (1, 2)), ("f16x2", 129, (1, 2)), ("f16x2", 48, (3, 9)), ("f16x2", 49, (3, 9)),
    ("f16x2", 300, (1, 4)), ("fp32", 257, (1, 2)), ("fp32", 300, (1, 9)), ("fp32", 301, (1, 3))])
def test_both_stages(k_prec, heights, replicas):
    need_gpu()
    el = _on_heights(s.graphene_plates(20, 15, 1, 30.0), heights)   # 2,400 sites: tables by height up to 300 heights
    assert el.n == 2400
    elyts = [s.ions_in_gap(el, 30 + 7 * r, seed=80 + r, dmin=2.0) for r in range(max(replicas))]
    ref = run_bvec(_ctx(el, "fp64"), elyts)
    some = np.arange(0, el.n, 97)
    sub = s.Electrodes(**{**el.__dict__, "xyz": el.xyz[some], "eta": el.eta[some], "group": el.group[some]})
    assert rel_l2(ref[0][some], o.bvec(sub, elyts[0])) <= 1e-11
    ctx = _ctx(el, k_prec)
    for m in replicas:
        b = run_bvec(ctx, elyts[:m])
        for r in range(m):
            assert rel_l2(b[r], ref[r]) <= 2e-6, (m, r)
