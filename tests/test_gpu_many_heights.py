"""b on electrodes whose sites hardly share heights, against the oracle (1e-11 relative L2 in FP64, 2e-6 in single
precision): numbers of heights at the edges of the k = 0 column's evaluation, and cells with more z harmonics than
the conversion to signed columns takes at a time."""
import numpy as np
import pytest

from gpu_util import dev, make_ctx, need_gpu, rel_l2, run_bvec, torch
from oracle import cpm_oracle as o
from paper_2203_15461_gb300 import systems as s

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-11, "fp32": 2e-6, "f16x2": 2e-6}


def _check(el, elyts, k_prec):
    ctx = make_ctx(el, k_prec=k_prec)
    ctx.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
    b = run_bvec(ctx, elyts)
    for r, e in enumerate(elyts):
        assert rel_l2(b[r], o.bvec(el, e)) <= TOL[k_prec], r


def _rough(n, box, seed, boundary):
    rng = np.random.default_rng(seed)
    base = s.au111_slab(seed_layers=1, nx=5, ny=4)
    xyz = rng.uniform(0.05, 0.95, (n, 3)) * box
    xyz[:, 2] = 0.1 * box[2] + np.linspace(0.0, 0.25, n) * box[2] + 0.01 * rng.uniform(size=n)
    return s.Electrodes(**{**base.__dict__, "xyz": xyz, "eta": np.full(n, 1.9), "group": (np.arange(n) % 2).astype(np.int32),
                           "box": box, "boundary": boundary})


@pytest.mark.parametrize("k_prec", ["fp32", "f16x2"])
@pytest.mark.parametrize("n", [255, 256, 257, 500])
def test_heights_of_the_first_column(n, k_prec):
    need_gpu()
    box = np.array([19.0, 23.0, 41.0])
    el = _rough(n, box, n, "slab")
    rng = np.random.default_rng(9)
    elyts = []
    for k in (30, 200, 1):
        x = rng.uniform(0.0, 1.0, (k, 3)) * box
        x[:, 2] = (0.45 + 0.4 * rng.uniform(size=k)) * box[2]
        elyts.append(s.Electrolyte(xyz=x, Q=rng.normal(size=k)))
    _check(el, elyts, k_prec)


@pytest.mark.parametrize("k_prec", ["fp64", "fp32", "f16x2"])
def test_many_harmonics(k_prec):
    need_gpu()
    box = np.array([13.0, 9.0, 900.0])
    el = _rough(48, box, 3, "3d")
    assert box[2] * el.kcut / (2.0 * np.pi) > 257
    rng = np.random.default_rng(2)
    elyts = [s.Electrolyte(xyz=rng.uniform(0.0, 1.0, (k, 3)) * box, Q=rng.normal(size=k)) for k in (40, 17)]
    _check(el, elyts, k_prec)
