"""Ensemble steps on a side stream whose members change buffers from call to
call, so that the step graph and the tables of its joined launches are made
anew each time: the members' results are those of their plans stepped alone,
bit for bit, and a call waits for its own earlier steps at most, not for other
work on the device.
"""
import numpy as np
import torch
import pytest

import paper_2405_13973_gb300 as pt
import workloads as W

pytestmark = pytest.mark.gpu


def members():
    spec = [("bf16x3", 300, 8), ("bf16x3", 900, 8), ("fp32", 500, 6), ("fp64", 400, 6), ("tf32x3", 700, 6)]
    crs = [W.ensemble_member(n, 0.5, seed=61 + k) for k, (_, n, _) in enumerate(spec)]
    plans = [pt.Plan(n, p=p, depth=2, precision=prec) for prec, n, p in spec]
    return crs, plans


def states(crs):
    return [pt.State.from_numpy(c["pos"], c["vel"], c["q"]) for c in crs]


def test_buffers_changing_on_a_side_stream():
    crs, plans = members()
    traps, dts = [pt.make_trap(c["trap"]) for c in crs], [c["dt"] for c in crs]
    alone = states(crs)
    for a in zip(plans, alone, traps, dts):
        a[0].step(a[1], a[2], None, a[3], 3)
    sets = [states(crs) for _ in range(3)]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    ens = pt.Ensemble(plans)
    for k in range(9):  # the sets in turn, one step each
        ens.step(sets[k % 3], traps, None, dts, 1, stream=side)
    ens.sync(stream=side)
    assert ens.joined_m2l() == 2
    ens.close()
    for st in sets:
        for s, a in zip(st, alone):
            assert torch.equal(s.pos(), a.pos()) and torch.equal(s.vel(), a.vel())
    for pl in plans:
        pl.close()


def test_a_new_graph_does_not_wait_for_other_work():
    crs, plans = members()
    traps, dts = [pt.make_trap(c["trap"]) for c in crs], [c["dt"] for c in crs]
    sets = [states(crs) for _ in range(3)]
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    ens = pt.Ensemble(plans)
    for st in sets[:2]:
        ens.step(st, traps, None, dts, 1, stream=side)
    ens.sync(stream=side)
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(other):
        torch.cuda._sleep(4_000_000_000)  # clock cycles: two seconds
        done.record()
    ens.step(sets[2], traps, None, dts, 1, stream=side)
    waited = done.query()
    ens.sync(stream=side)
    assert not waited
    torch.cuda.synchronize()
    ens.close()
    for pl in plans:
        pl.close()
