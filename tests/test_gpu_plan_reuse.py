"""A plan's results do not depend on what it computed before: after an
evaluation whose charges were NaN or overflowed the expansions, the next one
equals a new plan's, bit for bit, on every precision and schedule.

Depth 4 and an order whose coefficient count is no multiple of 32, so that the
expansions' rows have padding; the second crystal has fewer cells on the upper
levels, so that rows which held a parent's expansion hold a leaf's.
"""
import numpy as np
import pytest
import torch

import paper_2405_13973_gb300 as pt
import workloads as W

pytestmark = pytest.mark.gpu


def forces(plan, pos, q):
    E, phi = plan.forces(torch.tensor(np.ascontiguousarray(pos.T), device="cuda"),
                         torch.tensor(q, device="cuda"))
    return E.cpu().numpy(), phi.cpu().numpy()


@pytest.mark.parametrize("bad", [np.nan, 1e300])
@pytest.mark.parametrize("precision,schedule", [
    ("fp64", None), ("fp64", "tiles"), ("fp64", "pairs"), ("fp64", "rotation"), ("fp32", "tiles"),
    ("fp32", "pairs"), ("fp32", "rotation"), ("tf32x3", "tiles"), ("tf32x3", "pairs"),
    ("bf16x3", "tiles"), ("bf16x3", "pairs")])
def test_a_plan_recovers_from_nonfinite_expansions(precision, schedule, bad):
    n, p, depth = 3000, 12, 4
    ball = W.sphere_sweep(n, seed=9)["pos"]
    flat = ball[:900] * np.array([1.0, 1.0, 0.02])
    q = W.E_CHARGE * np.random.default_rng(3).choice([1.0, -1.0, 2.0], n)

    def plan():
        pl = pt.Plan(n, p=p, depth=depth, precision=precision)
        if schedule:
            pl.set_m2l_schedule(schedule)
        return pl

    used = plan()
    for pos in (ball, flat):
        try:
            forces(used, ball, q * bad)
        except pt.PenningError as err:
            assert err.status == pt.PT_ERR_NONFINITE
        E, phi = forces(used, pos, q[:len(pos)])
        new = plan()
        En, phin = forces(new, pos, q[:len(pos)])
        new.close()
        assert np.isfinite(En).all() and np.isfinite(phin).all()
        assert np.array_equal(E, En) and np.array_equal(phi, phin)
    used.close()
