"""FP64 b is linear in the charges over FP64's range: charges times 2^k give b times 2^k, to a few roundings (1e-13), also
where FP32 would overflow or underflow, and a charge that is not a number reaches every entry of b."""
import numpy as np
import pytest

from gpu_util import dev, make_ctx, need_gpu, rel_l2, run_bvec, torch
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu


def _b(el, elyts):
    ctx = make_ctx(el)
    ctx.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
    return run_bvec(ctx, elyts)


def _cloud(el, n):
    rng = np.random.default_rng(5)
    x = rng.uniform(0.0, 1.0, (n, 3)) * np.array([el.box[0], el.box[1], 18.0]) + np.array([0.0, 0.0, el.z_inner[0] + 3.0])
    return s.Electrolyte(xyz=x, Q=np.where(np.arange(n) < n // 2, 1.0, -1.0) * rng.uniform(0.2, 1.0, n))


@pytest.mark.parametrize("ions", [100, 4500])
@pytest.mark.parametrize("k", [-600, -140, 140, 600])
def test_fp64_b_scales(ions, k):
    need_gpu()
    el = s.au111_slab(seed_layers=1, nx=6, ny=6, gap=24.0)
    e = _cloud(el, ions)
    b1, bk = _b(el, [e, s.Electrolyte(xyz=e.xyz, Q=np.ldexp(e.Q, k))])
    assert np.isfinite(bk).all()
    assert rel_l2(np.ldexp(bk, -k), b1) <= 1e-13


@pytest.mark.parametrize("ions", [100, 4500])
def test_fp64_b_not_a_number(ions):
    need_gpu()
    el = s.au111_slab(seed_layers=1, nx=6, ny=6, gap=24.0)
    e = _cloud(el, ions)
    q = e.Q.copy()
    q[ions // 2] = np.nan
    b = _b(el, [e, s.Electrolyte(xyz=e.xyz, Q=q)])
    assert np.isfinite(b[0]).all() and np.isnan(b[1]).all()
