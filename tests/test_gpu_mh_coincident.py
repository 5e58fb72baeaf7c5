"""Metropolis-Hastings scans of crystals with ions at the same point, or so
close that their pair energy drowns the rest of a sum, against the oracle's
move after move: the same decisions, positions bit for bit.

A move's energy change has to be that of the positions at its turn: a pair
that an earlier move has parted adds nothing infinite, nor what is left of two
large terms that cancel.
"""
import math

import numpy as np
import pytest

import oracle
import paper_2405_13973_gb300 as pt
import workloads as W

pytestmark = pytest.mark.gpu


def place(kind, n):
    w = W.sphere_sweep(n, seed=4)
    pos, q = w["pos"].copy(), w["q"].copy()
    if kind == "pair":            # in different batches of moves
        pos[n - 1] = pos[3]
    elif kind == "opposite":      # unlike charges: the pair energy is -inf
        pos[9], q[9] = pos[0], -q[0]
    elif kind == "clump":
        pos[5:45] = pos[5]
    elif kind == "all":
        pos[:] = 0.0
    elif kind == "close":         # 60 pairs, pair energies of 1e16 k_B T
        pos[:60] = pos[60:120]
        pos[:60, 2] = 0.0
        pos[60:120, 2] = 1e-19
    elif kind == "nan":
        pos[7, 1] = np.nan
    return pos, q


@pytest.mark.parametrize("kind", ["pair", "opposite", "clump", "all", "close", "nan"])
@pytest.mark.parametrize("n", [126, 130, 300])
def test_mh_scans_with_coincident_ions_match_the_oracle(kind, n):
    pos, q = place(kind, n)
    trap = dict(W.crystal_sphere_1k(seed=11)["trap"], delta=0.02)
    t, scans = 3.7e-7, 2
    cs = (math.cos(trap["omega_r"] * t), math.sin(trap["omega_r"] * t))
    po, acc_o, _ = oracle.mh_scans(pos, q, trap, 10e-3, 1e-6, 17, 5, scans, cs)
    st = pt.State.from_numpy(pos, np.zeros_like(pos), q, t=t)
    acc, _ = pt.mh_scans(st, trap, 10e-3, 1e-6, 17, 5, scans)
    assert acc == acc_o
    assert np.array_equal(st.pos().cpu().numpy(), po, equal_nan=True)
