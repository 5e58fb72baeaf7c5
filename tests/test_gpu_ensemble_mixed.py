"""Ensembles whose members differ in precision, order and size (one ion, a crystal
without a far field, one beyond the one-launch tree, one with the larger
crystals' L2P): each member equals its plan stepped alone, bit for bit, and a
member's error is reported.
"""
import numpy as np
import pytest
import torch

import paper_2405_13973_gb300 as pt
import workloads as W

pytestmark = pytest.mark.gpu


def test_a_mixed_ensemble_equals_its_members_alone():
    spec = [("fp64", 1, 4), ("fp64", 700, 6), ("fp32", 2, 4), ("fp32", 900, 5), ("fp32", 17000, 4),
            ("tf32x3", 500, 6), ("tf32x3", 2600, 6), ("bf16x3", 3, 8), ("bf16x3", 400, 8),
            ("bf16x3", 2500, 5), ("bf16x3", 1500, 8), ("fp64", 2100, 8)]
    crs = [W.ensemble_member(n, 0.5, seed=31 + k) for k, (_, n, _) in enumerate(spec)]
    out = []
    for together in (True, False):
        plans = [pt.Plan(n, p=p, precision=prec) for prec, n, p in spec]
        states = [pt.State.from_numpy(c["pos"], c["vel"], c["q"]) for c in crs]
        traps = [pt.make_trap(c["trap"]) for c in crs]
        lasers = [pt.make_laser(c["beams"], seed=5 + k, gamma0=W.GAMMA0) for k, c in enumerate(crs)]
        dts = [c["dt"] for c in crs]
        if together:
            ens = pt.Ensemble(plans)
            ens.step(states, traps, lasers, dts, 4)
            ens.sync()
            ens.close()
        else:
            for a in zip(plans, states, traps, lasers, dts):
                a[0].step(*a[1:], 4)
        torch.cuda.synchronize()
        out.append([(s.pos().cpu().numpy(), s.vel().cpu().numpy()) for s in states])
        for pl in plans:
            pl.close()
    for k, ((xm, vm), (xa, va)) in enumerate(zip(*out)):
        assert np.array_equal(xm, xa) and np.array_equal(vm, va), spec[k]


def test_an_ensemble_reports_a_members_error():
    crs = [W.ensemble_member(n, 0.5, seed=3 + n) for n in (100, 300, 200)]
    crs[1]["pos"][7, 2] = np.nan
    plans = [pt.Plan(len(c["q"]), p=6, precision="bf16x3", depth=2) for c in crs]
    states = [pt.State.from_numpy(c["pos"], c["vel"], c["q"]) for c in crs]
    traps = [pt.make_trap(c["trap"]) for c in crs]
    ens = pt.Ensemble(plans)
    with pytest.raises(pt.PenningError) as err:
        ens.step(states, traps, None, [c["dt"] for c in crs], 2)
        ens.sync()
    assert err.value.status == pt.PT_ERR_NONFINITE
    ens.sync()  # reported once
    assert np.isfinite(states[0].pos().cpu().numpy()).all()
    ens.close()
    for pl in plans:
        pl.close()
