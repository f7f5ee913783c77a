"""P3M charge assignment and the planes left out: b against the oracle's P3M (1e-12 in FP64, 2e-6 in single precision,
as the other P3M tests) with charges above and below 2 e, more charges at one place than are added between two carries,
one replica more than a pair, an empty replica, and meshes with one and several bricks per axis."""
import numpy as np
import pytest

from gpu_util import dev, make_ctx, need_gpu, rel_l2, run_bvec, torch
from oracle import cpm_oracle as o
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k_prec,tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("mesh,order", [((32, 32, 64), 7), ((64, 64, 64), 5), ((8, 128, 32), 3), ((64, 16, 128), 6)])
def test_p3m_assignment(mesh, order, k_prec, tol):
    need_gpu()
    base = s.au111_slab(seed_layers=1, nx=5, ny=6, gap=24.0)
    el = s.Electrodes(**{**base.__dict__, "p3m_mesh": mesh, "p3m_order": order})
    rng = np.random.default_rng(12)
    zc = 0.5 * (el.z_inner[0] + el.z_inner[1])

    def cloud(n, spread, qmax):
        x = np.column_stack([rng.uniform(0, el.box[0], n), rng.uniform(0, el.box[1], n), zc + rng.uniform(-spread, spread, n)])
        return s.Electrolyte(xyz=x, Q=rng.uniform(-qmax, qmax, n))

    crowd = cloud(2600, 0.02, 0.8)                      # one chunk after the other in the same planes
    crowd.xyz[:, :2] = crowd.xyz[0, :2] + rng.uniform(-0.05, 0.05, (2600, 2))
    elyts = [crowd, cloud(90, 6.0, 40.0), s.Electrolyte(xyz=np.zeros((0, 3)), Q=np.zeros(0)), cloud(513, 8.0, 1.9),
             cloud(1, 1.0, 1.0)]
    ctx = make_ctx(el, k_prec=k_prec)
    ctx.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
    b = run_bvec(ctx, elyts)
    for r, e in enumerate(elyts):
        if e.n == 0:
            # the rounding of the partner in the shared mesh, which has the partner's relative accuracy
            assert np.abs(b[r]).max() <= tol * np.abs(b[r + 1]).max()
        else:
            assert rel_l2(b[r], o.bvec(el, e)) <= tol, r


@pytest.mark.parametrize("k_prec,tol", [("fp64", 1e-12), ("fp32", 2e-6)])
@pytest.mark.parametrize("sites_per_height", [1, 7, 8, 30])
def test_p3m_shared_and_single_heights(sites_per_height, k_prec, tol):
    """Every site on a height of its own (interpolation over the mesh) to whole layers (one plane per height)."""
    need_gpu()
    base = s.au111_slab(seed_layers=2, nx=5, ny=6, gap=24.0)
    first = (np.arange(base.n) // sites_per_height) * sites_per_height
    xyz = base.xyz.copy()
    xyz[:, 2] = (base.xyz[:, 2] + 0.2 * np.sin(first * 1.7 + 0.3))[first]
    el = s.Electrodes(**{**base.__dict__, "xyz": xyz, "p3m_mesh": (32, 16, 64), "p3m_order": 5})
    elyts = [s.ions_in_gap(el, 40 + 9 * r, seed=60 + r, dmin=2.0) for r in range(3)]
    ctx = make_ctx(el, k_prec=k_prec)
    ctx.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
    b = run_bvec(ctx, elyts)
    for r, e in enumerate(elyts):
        assert rel_l2(b[r], o.bvec(el, e)) <= tol, r


@pytest.mark.parametrize("k_prec,tol", [("fp64", 1e-12), ("fp32", 2e-6)])
def test_p3m_brick_lists(k_prec, tol):
    """Enough charges for several splits, bricks on both sides of every face of the cell, and the same bits each time."""
    need_gpu()
    base = s.au111_slab(seed_layers=1, nx=5, ny=6, gap=24.0)
    el = s.Electrodes(**{**base.__dict__, "p3m_mesh": (64, 32, 64), "p3m_order": 7})
    rng = np.random.default_rng(21)

    def cloud(n):
        x = rng.uniform(-0.3, 1.3, (n, 3)) * np.array([el.box[0], el.box[1], 0.0])
        x[:, 2] = rng.uniform(el.z_inner[0] + 3.0, el.z_inner[1] - 3.0, n)
        return s.Electrolyte(xyz=x, Q=rng.uniform(-1.0, 1.0, n))

    elyts = [cloud(5000), cloud(1537), cloud(4608)]
    ctx = make_ctx(el, k_prec=k_prec)
    ctx.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
    b = run_bvec(ctx, elyts)
    for r, e in enumerate(elyts):
        assert rel_l2(b[r], o.bvec(el, e)) <= tol, r
    for _ in range(3):
        assert np.array_equal(run_bvec(ctx, elyts), b)
