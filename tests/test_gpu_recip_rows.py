"""Reciprocal-space b in the real product basis: the height-wise site stage and the general one.

Against the oracle at the tolerances of the other b tests (1e-11 relative L2 in FP64, 2e-6 on the single-precision
paths): charge counts at the edges of the kernels' charge ranges, replica counts at the edges of the site
stage's replica groups, odd lattices, and electrodes whose sites have all different heights (general stage) or
share them at exactly the limit between the two stages.
"""
import numpy as np
import pytest

from gpu_util import dev, make_ctx, need_gpu, rel_l2, run_bvec, torch
from oracle import cpm_oracle as o
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-11, "fp32": 2e-6, "f16x2": 2e-6}


def _heights(el, sites_per_height):
    """The same sites with heights changed by up to 0.2 A, sites_per_height of them on each."""
    z = el.xyz[:, 2] + 0.2 * np.sin(np.arange(el.n) // sites_per_height * 1.7 + 0.3)
    first = (np.arange(el.n) // sites_per_height) * sites_per_height
    xyz = el.xyz.copy()
    xyz[:, 2] = z[first]
    return s.Electrodes(**{**el.__dict__, "xyz": xyz})


def _b(el, elyts, k_prec):
    ctx = make_ctx(el, k_prec=k_prec)
    ctx.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
    return run_bvec(ctx, elyts)


@pytest.mark.parametrize("k_prec", ["fp64", "fp32", "f16x2"])
@pytest.mark.parametrize("n_ions", [(1,), (2, 64), (16, 65, 17), (63, 3, 128, 100, 1), (31,) * 9])
def test_charge_and_replica_counts(k_prec, n_ions):
    need_gpu()
    el = s.au111_slab(seed_layers=1, nx=5, ny=6, gap=24.0)
    elyts = [s.ions_in_gap(el, k, seed=40 + r, dmin=1.5) for r, k in enumerate(n_ions)]
    b = _b(el, elyts, k_prec)
    for r, e in enumerate(elyts):
        assert rel_l2(b[r], o.bvec(el, e)) <= TOL[k_prec], r


@pytest.mark.parametrize("k_prec", ["fp64", "fp32", "f16x2"])
@pytest.mark.parametrize("sites_per_height", [1, 7, 8, 30])
def test_shared_and_single_heights(k_prec, sites_per_height):
    need_gpu()
    el = _heights(s.au111_slab(seed_layers=2, nx=5, ny=4), sites_per_height)
    elyts = [s.ions_in_gap(el, 40 + 9 * r, seed=60 + r, dmin=2.0) for r in range(3)]
    b = _b(el, elyts, k_prec)
    for r, e in enumerate(elyts):
        assert rel_l2(b[r], o.bvec(el, e)) <= TOL[k_prec], r


@pytest.mark.parametrize("k_prec", ["fp64", "fp32", "f16x2"])
@pytest.mark.parametrize("boundary,box", [("3d", (23.0, 29.0, 37.0)), ("slab", (70.0, 19.0, 90.0)), ("wire", (75.0, 66.0, 11.0))])
def test_odd_boxes(k_prec, boundary, box):
    """Boxes with very different harmonic counts per axis (also more x and y harmonics than fit one tile)."""
    need_gpu()
    rng = np.random.default_rng(5)
    base = s.au111_slab(seed_layers=1, nx=5, ny=4)
    n, box = 48, np.array(box)
    xyz = rng.uniform(0.05, 0.95, (n, 3)) * box
    xyz[:, 2] = np.repeat(np.linspace(0.1, 0.8, 4) * box[2], n // 4)
    el = s.Electrodes(**{**base.__dict__, "xyz": xyz, "eta": np.full(n, 1.9), "group": (np.arange(n) % 2).astype(np.int32),
                         "box": box, "boundary": boundary})
    ely = [s.Electrolyte(xyz=rng.uniform(0.0, 1.0, (k, 3)) * box, Q=rng.normal(size=k)) for k in (70, 33)]
    b = _b(el, ely, k_prec)
    for r, e in enumerate(ely):
        assert rel_l2(b[r], o.bvec(el, e)) <= TOL[k_prec], r
