"""FP64 structure factor by integer products: b within 1e-11 (relative L2) of the oracle, as the other FP64 b tests, with
charge counts at the edges of the steps (32) and of the ranges (480), charges from 1e-6 to 700 e in one replica, heights
shared and not shared, boxes with one and with several tiles of pairs and harmonics, and against the FP64 pipe's own
sum on the same charges (few replicas take that path, many this one)."""
import numpy as np
import pytest

from gpu_util import dev, make_ctx, need_gpu, rel_l2, run_bvec, torch
from oracle import cpm_oracle as o
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu


def _b(el, elyts):
    ctx = make_ctx(el)
    ctx.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
    return run_bvec(ctx, elyts)


def _cloud(rng, el, n, q):
    z0, z1 = float(el.xyz[:, 2].min()) + 3.0, float(el.xyz[:, 2].max()) - 3.0
    lo, hi = min(z0, z1), max(z0, z1)
    return s.Electrolyte(xyz=np.column_stack([rng.uniform(0, el.box[0], n), rng.uniform(0, el.box[1], n),
                                              rng.uniform(lo, hi, n)]), Q=q)


@pytest.mark.parametrize("counts", [(5000,), (479, 480, 481, 4000), (31, 32, 33, 3900, 1), (2900, 2911)])
def test_rows64_counts(counts):
    need_gpu()
    el = s.au111_slab(seed_layers=1, nx=6, ny=6, gap=24.0)
    rng = np.random.default_rng(len(counts))
    elyts = [_cloud(rng, el, n, rng.normal(size=n)) for n in counts]
    b = _b(el, elyts)
    for r, e in enumerate(elyts):
        assert rel_l2(b[r], o.bvec(el, e)) <= 1e-11, r


@pytest.mark.parametrize("scale", [1e-6, 1.0, 512.0, 700.0])
def test_rows64_charge_range(scale):
    """The largest charge a power of two and not, the others down to 1e-6 of it."""
    need_gpu()
    el = s.au111_slab(seed_layers=2, nx=5, ny=6, gap=24.0)
    rng = np.random.default_rng(4)
    q = scale * 10.0 ** rng.uniform(-6.0, 0.0, 4500) * np.where(rng.random(4500) < 0.5, 1.0, -1.0)
    q[7] = scale
    e = _cloud(rng, el, 4500, q)
    assert rel_l2(_b(el, [e])[0], o.bvec(el, e)) <= 1e-11


@pytest.mark.parametrize("boundary,box", [("3d", (23.0, 29.0, 37.0)), ("slab", (60.0, 19.0, 90.0)), ("wire", (55.0, 50.0, 11.0))])
@pytest.mark.parametrize("shared", [True, False])
def test_rows64_boxes(boundary, box, shared):
    need_gpu()
    rng = np.random.default_rng(6)
    base = s.au111_slab(seed_layers=1, nx=5, ny=4)
    n, box = 48, np.array(box)
    xyz = rng.uniform(0.05, 0.95, (n, 3)) * box
    if shared:
        xyz[:, 2] = np.repeat(np.linspace(0.1, 0.8, 4) * box[2], n // 4)
    el = s.Electrodes(**{**base.__dict__, "xyz": xyz, "eta": np.full(n, 1.9), "group": (np.arange(n) % 2).astype(np.int32),
                         "box": box, "boundary": boundary})
    elyts = [s.Electrolyte(xyz=rng.uniform(0.0, 1.0, (k, 3)) * box, Q=rng.normal(size=k)) for k in (1501, 2017)]
    b = _b(el, elyts)
    for r, e in enumerate(elyts):
        assert rel_l2(b[r], o.bvec(el, e)) <= 1e-11, r


def test_rows64_against_fp64_pipe():
    """40 replicas of 100 ions in one call (integer products) and one by one (FP64 multiply-adds)."""
    need_gpu()
    el = s.au111_slab()
    elyts = [s.ions_in_gap(el, 100, seed=300 + r) for r in range(40)]
    many = _b(el, elyts)
    for r in (0, 17, 39):
        assert rel_l2(many[r], _b(el, [elyts[r]])[0]) <= 1e-13
