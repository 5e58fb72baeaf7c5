"""Metropolis-Hastings scans at the edges of a batch of 128 moves and of the
scratch kept for up to 4,096 ions, against the oracle, as in the scan tests:
the same decisions and positions bit for bit, the energy to 1e-9."""
import math

import numpy as np
import pytest

import oracle
import paper_2405_13973_gb300 as pt
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,scans", [(1, 5), (2, 3), (127, 2), (128, 2), (129, 2), (257, 1),
                                     (4096, 1), (4097, 1)])
def test_mh_batch_edges_match_the_oracle(n, scans):
    w = W.sphere_sweep(max(n, 2), seed=4)
    pos, q = w["pos"][:n].copy(), w["q"][:n].copy()
    trap = dict(W.crystal_sphere_1k(seed=11)["trap"], delta=0.02)
    t = 3.7e-7
    cs = (math.cos(trap["omega_r"] * t), math.sin(trap["omega_r"] * t))
    po, acc_o, de_o = oracle.mh_scans(pos, q, trap, 10e-3, 1e-6, 17, 5, scans, cs)
    st = pt.State.from_numpy(pos, np.zeros_like(pos), q, t=t)
    acc, de = pt.mh_scans(st, trap, 10e-3, 1e-6, 17, 5, scans)
    assert acc == acc_o
    assert np.array_equal(st.pos().cpu().numpy(), po)
    assert abs(de - de_o) <= 1e-9 * abs(de_o)
