"""P2M and L2P with a thread per ion (larger crystals) against the kernels that
smaller crystals take: the same charges, with ions of zero charge added inside
the crystal until its size crosses a kernel's line, have the same field.

The depth is given, so the charged ions keep their cells; the added ions split
the windows of sorted slots elsewhere, open leaves that hold no charge and, at
depth 2, fill leaves beyond one pass of a block.  Bounds: rounding of sums of
some 1e4 terms, sqrt(1e4) u at most for the relative error of the whole field;
1e-12 for u = 1.1e-16 (1e-14 each over the chain of P2M, shifts, M2L, L2P and
the near field, whose sums cancel by up to 10), and 4e-6 in FP32 (u = 6e-8; the
reordered near field alone has a bound of 2e-6).
"""
import numpy as np
import pytest
import torch

import paper_2405_13973_gb300 as pt

pytestmark = pytest.mark.gpu

N0 = 7000


def crystal(seed):
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((N0, 3))
    u *= (rng.random(N0) ** (1 / 3) / np.linalg.norm(u, axis=1))[:, None]
    return u * np.array([1e-3, 8e-4, 3e-4]), rng.choice([1.0, 2.0], N0) * 1.602176634e-19


@pytest.fixture(scope="module")
def base():
    return crystal(77)


def field(pos, q, precision, p, depth):
    plan = pt.Plan(len(pos), p=p, depth=depth, precision=precision)
    E, phi = plan.forces(torch.tensor(pos.T.copy(), device="cuda"), torch.tensor(q, device="cuda"))
    E, phi = E.cpu().numpy()[:, :N0], phi.cpu().numpy()[:N0]
    plan.close()
    return E, phi


@pytest.mark.parametrize("precision,p,depth", [
    ("fp64", 2, 2), ("fp64", 7, 4), ("fp64", 12, 3), ("fp64", 16, 2),
    ("fp32", 2, 3), ("fp32", 7, 2), ("fp32", 8, 4), ("fp32", 9, 3), ("fp32", 14, 3),
    ("fp32", 15, 4), ("fp32", 16, 3)])
def test_field_across_the_kernels_lines(base, precision, p, depth):
    pos, q = base
    i = np.arange(12000)  # midpoints of two different ions each
    extra = 0.5 * (pos[i % N0] + pos[(i + 1 + i // N0) % N0])
    E0, phi0 = field(pos, q, precision, p, depth)
    tol = 1e-12 if precision == "fp64" else 4e-6
    for n in ((7168, 10239, 10240, 10301) if precision == "fp64" else (16383, 16384, 16497)):
        k = n - N0
        E, phi = field(np.concatenate([pos, extra[:k]]), np.concatenate([q, np.zeros(k)]),
                       precision, p, depth)
        assert np.linalg.norm(E - E0) < tol * np.linalg.norm(E0), n
        assert np.linalg.norm(phi - phi0) < tol * np.linalg.norm(phi0), n
