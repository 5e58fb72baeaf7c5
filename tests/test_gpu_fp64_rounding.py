"""Rounding of the default FP64 translations (tensor-core digit products)
against the same truncated expansions in long double: no larger than that of
the FP64 multiply-add schedules.

The reference is the field of a few leaves, level by level: multipoles of the
source cells from their ions, Eq. FMM_local, the local expansions of the leaf
and its ancestors at the ions (M2M and L2L do not change a truncated
expansion's values).  The leaves' errors are a sample of a few dozen values:
twice the larger multiply-add error is allowed.
"""
import numpy as np
import pytest
import torch

import paper_2405_13973_gb300 as pt
import workloads as W

pytestmark = pytest.mark.gpu
LD, CLD = np.longdouble, np.clongdouble


def harmonics(p, u, irregular=False):
    """X[n, m + p] of points u (3, k): Y_n^m, or Th_n^m."""
    w, z, r2 = u[0] + CLD(1j) * u[1], u[2].astype(CLD), (u * u).sum(0)
    X = np.zeros((p + 1, 2 * p + 1, u.shape[1]), CLD)
    i2 = 1 / r2
    d = np.sqrt(i2).astype(CLD) if irregular else np.ones(u.shape[1], CLD)
    for m in range(p + 1):
        if m > 0:
            d = d * w * ((2 * m - 1) * i2 if irregular else 1 / LD(2 * m))
        X[m, p + m] = d
        if m < p:
            X[m + 1, p + m] = z * d * ((2 * m + 1) * i2 if irregular else 1)
        for n in range(m + 2, p + 1):
            a, b = X[n - 1, p + m], X[n - 2, p + m]
            X[n, p + m] = (((2 * n - 1) * z * a - ((n - 1) ** 2 - m * m) * b) * i2 if irregular else
                           ((2 * n - 1) * z * a - r2 * b) / LD((n + m) * (n - m)))
    for m in range(1, p + 1):
        X[:, p - m] = (-1) ** m * X[:, p + m].conj()
    return X


def coordinates(key, depth):
    return np.array([sum(((key >> (3 * b + 2 - a)) & 1) << b for b in range(depth)) for a in range(3)])


def reference(pos, q, key, root, depth, p, leaves):
    """(ions, E (3, .)) of the given leaf keys."""
    x = (pos.astype(LD) - np.array(root[:3], LD)[:, None]) / LD(root[3])  # unit cube
    ions = np.nonzero(np.isin(key, leaves))[0]
    E = np.zeros((3, len(pos[0])), LD)
    offs = [o for o in np.ndindex(7, 7, 7) if max(abs(c - 3) for c in o) > 1]
    for l in range(2, depth + 1):
        cell = coordinates(key >> (3 * (depth - l)), l)
        u = x * 2 ** l - cell - LD(0.5)
        for t in np.unique(leaves >> (3 * (depth - l))):
            c = coordinates(np.array([t]), l)[:, 0]
            L = np.zeros((p + 1, 2 * p + 1), CLD)
            for o in offs:
                o = np.array(o) - 3
                if (abs(((c - o) >> 1) - (c >> 1)) > 1).any():
                    continue
                src = (cell == (c - o)[:, None]).all(0)
                if not src.any():
                    continue
                M = (q[src] * harmonics(p, u[:, src]).conj()).sum(-1)
                Th = harmonics(2 * p, o.astype(LD)[:, None], True)[:, :, 0]
                for a in range(p + 1):
                    for b in range(-a, a + 1):
                        L[a, p + b] += (-1) ** a * (M * Th[a:a + p + 1, p + b:3 * p + b + 1]).sum()
            at = np.nonzero((key >> (3 * (depth - l)) == t) & np.isin(key, leaves))[0]
            Y = np.zeros((p + 1, 2 * p + 3, len(at)), CLD)
            Y[1:, 1:-1] = harmonics(p, u[:, at])[:-1]          # Y_{n-1}^m
            up, down, mid = -Y[:, 2:], Y[:, :-2], Y[:, 1:-1]   # d/dx + i d/dy, d/dx - i d/dy, d/dz
            # the real part of a sum over every m; conj(Y) is what L meets
            for k, dY in enumerate(((up + down) / 2, (up - down) / CLD(2j), mid)):
                E[k, at] -= (L[:, :, None] * dY.conj()).sum((0, 1)).real * LD(4) ** l
    ke = LD(1 / (4 * np.pi * 8.8541878128e-12))
    return ions, ke / LD(root[3]) ** 2 * E[:, ions]


@pytest.mark.parametrize("n,p,depth,picked", [(4000, 4, 4, 10), (2500, 8, 3, 6), (2500, 12, 3, 2)])
def test_fp64_default_rounds_no_more_than_multiply_adds(n, p, depth, picked):
    w = W.sphere_sweep(n, seed=21)
    pos, q = np.ascontiguousarray(w["pos"].T), w["q"]
    out = []
    for schedule in (None, "pairs", "rotation"):
        plan = pt.Plan(n, p=p, depth=depth, precision="fp64")
        if schedule:
            plan.set_m2l_schedule(schedule)
        plan.set_phases(pt.PT_PHASE_FAR)
        E, _ = plan.forces(torch.tensor(pos, device="cuda"), torch.tensor(q, device="cuda"))
        root, _, key = plan.tree_info(n)
        out.append(E.cpu().numpy())
        plan.close()
    key = key.cpu().numpy().astype(np.int64)
    leaves = np.random.default_rng(5).choice(np.unique(key), picked, replace=False)
    ions, Er = reference(pos, q, key, root, depth, p, leaves)
    err = [float(np.linalg.norm((E[:, ions] - Er).astype(np.float64)) /
                 np.linalg.norm(Er.astype(np.float64))) for E in out]
    assert max(err) < 1e-12  # the reference is the same expansion
    assert err[0] < 2 * max(err[1:]), err
