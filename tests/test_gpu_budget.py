"""A budget with no room for the partial sums of the fast plans: the calls take plans of fewer sums instead of refusing,
with the same b and q (the tolerances of the precisions), and refuse when nothing fits."""
import numpy as np
import pytest

from gpu_util import dev, make_ctx, need_gpu, rel_l2, run_bvec, run_update, torch
from paper_2203_15461_gb300 import systems as s
from paper_2203_15461_gb300.cpm import CPMError

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "fp32": 2e-6, "f16x2": 2e-6}


# the last: the share of the scratch that the budget has room for (with P3M the charges themselves, their cell list and
# one mesh are most of it)
@pytest.mark.parametrize("k_prec,m,ions,p3m,share", [
    ("fp64", 1, 100, False, 0.6), ("fp64", 1, 1500, False, 0.6), ("fp64", 9, 400, False, 0.6), ("fp32", 1, 1000, False, 0.6),
    ("fp32", 8, 200, False, 0.6), ("f16x2", 1, 3000, False, 0.6), ("fp32", 4, 3500, True, 0.6), ("fp64", 2, 3500, True, 0.8)])
def test_b(k_prec, m, ions, p3m, share):
    need_gpu()
    el = s.au111_slab(seed_layers=2, nx=6, ny=6, gap=30.0)
    el = s.with_p3m(el) if p3m else el
    rng = np.random.default_rng(ions)
    elyts = []
    for r in range(m):
        x = rng.uniform(0.0, 1.0, (ions, 3)) * np.array([el.box[0], el.box[1], 20.0]) + [0.0, 0.0, el.z_inner[0] + 5.0]
        elyts.append(s.Electrolyte(xyz=x, Q=rng.normal(size=ions)))

    def ctx(budget):
        c = make_ctx(el, k_prec=k_prec, s_prec="fp32", hbm_budget=budget)
        c.cpm_prepare(dev(el.xyz), dev(el.eta), dev(el.group, torch.int32), el.n_groups)
        return c
    full = ctx(0)
    held = full.cpm_device_bytes()
    ref = run_bvec(full, elyts)
    need = full.cpm_device_bytes()
    for room in (need - 4096, held + int((need - held) * share)):
        b = run_bvec(ctx(room), elyts)
        for r in range(m):
            assert rel_l2(b[r], ref[r]) <= TOL[k_prec], (room, r)
    with pytest.raises(CPMError):
        run_bvec(ctx(held + 4096), elyts)


def test_fp64_update():
    need_gpu()
    el = s.graphene_plates(8, 5, 2, 30.0)
    rng = np.random.default_rng(1)
    b, psi = rng.normal(size=(24, el.n)), np.array([0.0, 1.0])

    def ctx(budget):
        return make_ctx(el, k_prec="fp32", hbm_budget=budget).setup(el)
    full = ctx(0)
    held = full.cpm_device_bytes()
    q, _ = run_update(full, psi, b)
    need = full.cpm_device_bytes()
    for room in (need - 4096, held + (need - held) // 4):
        assert rel_l2(run_update(ctx(room), psi, b)[0], q) <= 1e-12
    with pytest.raises(CPMError):
        run_update(ctx(held + 4096), psi, b)
