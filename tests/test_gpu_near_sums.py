"""FP64 near field: large pair terms that cancel leave the small ones whole.

One leaf (depth 0), coordinates that are multiples of a power of two, so that
every separation is exact: two charges of 1e9 e and opposite sign at equal
distances from a target add up to nothing.  Up to 11 ions every source is a
chunk of its own (128 threads, chunks x targets), and with the rounding
carried along (compensated sums between chunks) what is left is off by a few
roundings of the small terms, below 1e-14 of them; without, by roundings of
the large terms, 1e9 x 1e-16.
"""
import numpy as np
import pytest
import torch

import paper_2405_13973_gb300 as pt
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 6, 8, 11])
@pytest.mark.parametrize("want_phi", [True, False])
def test_cancelling_pairs_leave_the_small_terms(n, want_phi):
    rng = np.random.default_rng(n)
    pos = rng.integers(-31, 32, (n, 3)) / 64.0
    pos[0], pos[1] = (-0.5, -0.5, -0.5), (0.5, 0.5, 0.5)   # the root cube: side 1
    t, a, b = 2, 3, n - 1
    pos[t] = 0.0
    pos[a], pos[b] = (0.25, 0.125, 0.0), (-0.25, 0.125, 0.0)
    q = rng.integers(1, 4, n) * W.E_CHARGE
    q[a], q[b] = 1e9 * W.E_CHARGE, -1e9 * W.E_CHARGE
    s = 2.0 ** -10
    plan = pt.Plan(n, p=4, depth=0, precision="fp64")
    E, phi = plan.forces(torch.tensor(np.ascontiguousarray(pos.T) * s, device="cuda"),
                         torch.tensor(q, device="cuda"), want_phi=want_phi)
    plan.close()
    r = (pos[t] - np.delete(pos, t, 0)).astype(np.longdouble) * s
    w = np.delete(q, t) / np.sqrt((r * r).sum(1))
    ke = 1.0 / (4.0 * np.pi * 8.8541878128e-12)
    small = np.delete(np.abs(q) < 1e6 * W.E_CHARGE, t)
    # the large pair cancels in phi, and in E_y and E_z
    e = (w / (r * r).sum(1))[:, None] * r
    if want_phi:
        assert abs(float(phi[t]) - ke * w.sum()) < 1e-14 * ke * abs(w[small]).sum()
    for k in (1, 2):
        assert abs(float(E[k, t]) - ke * e[:, k].sum()) < 1e-14 * ke * abs(e[small, k]).sum()
