"""FP64 real-space sum and S product: b within 1e-11 (relative L2, as the other FP64 b tests) and q within 1e-10 of the
oracle where the pair tables, the image shifts and the row loops can go wrong.

Charges on top of a site and inside the Gaussian cores, two very different widths, charges at the cut-off, cut-offs longer
than the box, many charges in one cell, and site counts around the column pairs and replica groups of the S product.
"""
import numpy as np
import pytest

from gpu_util import dev, make_ctx, need_gpu, rel_l2, run_bvec, run_update, torch
from oracle import cpm_oracle as o
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu


def _slab(nx=5, ny=4, layers=1, eta=None, **kw):
    el = s.au111_slab(seed_layers=layers, nx=nx, ny=ny, **kw)
    return el if eta is None else s.Electrodes(**{**el.__dict__, "eta": np.resize(np.asarray(eta, float), el.n)})


def _b(el, elyts):
    """b alone: no elastance matrix, so any splitting and cut-off will do."""
    ctx = make_ctx(el)
    ctx.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
    return run_bvec(ctx, elyts)


@pytest.mark.parametrize("eta", [(1.979,), (0.6, 6.0), (0.45,)], ids=["au", "two", "wide"])
@pytest.mark.parametrize("rcut", [3.0, 12.0, 29.0])
def test_real64_pairs(eta, rcut):
    """Distances from nearly zero to past the cut-off of one site, exact multiples of the interval edges among them."""
    need_gpu()
    el = _slab(eta=eta, rcut=rcut)
    r = np.concatenate([[1e-3, 0.0625, 0.25, 0.5, 1.0, 2.0, rcut * (1 - 1e-13), rcut * (1 + 1e-13)],
                        np.linspace(0.01, min(rcut, 14.0), 53)])
    u = np.random.default_rng(3).normal(size=(len(r), 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    at = el.xyz[np.arange(len(r)) % el.n]
    ely = s.Electrolyte(xyz=at + r[:, None] * u, Q=np.where(np.arange(len(r)) % 2 == 0, 1.0, -0.7))
    # a pair at the cut-off to 1e-13 counts on one side of it or the other: leave those two out of the oracle's share
    ely = s.Electrolyte(xyz=np.delete(ely.xyz, [6, 7], axis=0), Q=np.delete(ely.Q, [6, 7]))
    b = _b(el, [ely])
    assert rel_l2(b[0], o.bvec(el, ely)) <= 1e-11


def test_real64_coincident():
    """A charge on a site: the limit of the pair function, where the oracle's formula is 0 / 0.  b at the site then differs
    from b with the charge 1e-6 A away by terms of second order (1e-12)."""
    need_gpu()
    el = _slab()
    b = [_b(el, [s.Electrolyte(xyz=el.xyz[2:3] + np.array([[d, 0.0, 0.0]]), Q=np.ones(1))])[0] for d in (0.0, 1e-9, 1e-6)]
    assert abs(b[0][2] - b[2][2]) <= 1e-10 * abs(b[2][2])
    assert abs(b[1][2] - b[2][2]) <= 1e-10 * abs(b[2][2])


def test_real64_crowded_cell_and_far_images():
    """200 charges within 2 A of one point and charges several periods outside the cell."""
    need_gpu()
    el = _slab(nx=5, ny=4, layers=2)
    rng = np.random.default_rng(8)
    xyz = np.concatenate([el.xyz[3] + np.array([0.0, 0.0, 3.0]) + rng.uniform(-1.0, 1.0, (200, 3)),
                          rng.uniform(0, 1, (30, 3)) * el.box * 0.3 + np.array([3.0, -2.0, 0.0]) * el.box])
    ely = s.Electrolyte(xyz=xyz, Q=rng.normal(size=len(xyz)))
    b = _b(el, [ely])
    assert rel_l2(b[0], o.bvec(el, ely)) <= 1e-11


@pytest.mark.parametrize("nx,m", [(5, 1), (5, 2), (6, 3), (7, 5), (9, 8), (5, 9)])
def test_fp64_update_sizes(nx, m):
    """40 to 72 sites, less one for an odd count: every replica group and both column widths of the S product."""
    need_gpu()
    el = _slab(nx=nx, ny=4)
    if m % 2:
        keep = np.arange(el.n - 1)
        el = s.Electrodes(**{**el.__dict__, "xyz": el.xyz[keep], "eta": el.eta[keep], "group": el.group[keep]})
    ctx = make_ctx(el).setup(el)
    elyts = [s.ions_in_gap(el, 20 + r, seed=90 + r) for r in range(m)]
    psi = np.array([0.0, 1.0])
    b = run_bvec(ctx, elyts)
    q, qt = run_update(ctx, psi, b)
    S = o.capacitance_matrix(o.assemble_A(el))
    for r, e in enumerate(elyts):
        assert rel_l2(q[r], o.charges(S, el, psi, o.bvec(el, e))) <= 1e-10
    assert np.abs(qt).max() <= 1e-12
