"""FP64 and FP32 translations of the default schedules (tensor-core digit
slices; packed FP32 tiles) against the CUDA-core schedules that an explicit
choice selects, and against each other.

Bounds, relative to the whole far field: the sums of one target run over at
most 189 (p + 1)^2 < 6e4 products in three stages (M2M, M2L, L2L); FP64
rounding of such sums, 3 x sqrt(6e4) u, is below 1e-13 (u = 1.1e-16) and a
slice product is exact, so 1e-12, the bound between the CUDA-core schedules
themselves.  FP32 against FP64 of the same tree: 3 x sqrt(6e4) u = 4.4e-5 for
errors that all add up, 2e-6 as between the FP32 schedules for errors that do
not, twice that with the rounding of the positions and of L2P.
"""
import numpy as np
import pytest
import torch

import paper_2405_13973_gb300 as pt
import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda"


def rel(a, b):
    m = np.abs(b).max()
    return float(np.linalg.norm((a - b) / m) / np.linalg.norm(b / m))


def far(pos, q, p, depth, precision, schedule=None, n_max=None):
    plan = pt.Plan(n_max or len(q), p=p, depth=depth, precision=precision)
    if schedule:
        plan.set_m2l_schedule(schedule)
    plan.set_phases(pt.PT_PHASE_FAR)
    E, phi = plan.forces(torch.tensor(np.ascontiguousarray(pos.T), device=DEV),
                         torch.tensor(q, device=DEV))
    out = E.cpu().numpy(), phi.cpu().numpy()
    plan.close()
    return out


def charges(kind, pos):
    rng = np.random.default_rng(3)
    q = W.E_CHARGE * rng.choice([1.0, -1.0, 2.0], len(pos))
    if kind == "zeros":     # a half space without charge: zero expansions
        return np.where(pos[:, 0] > 0, q, 0.0)
    if kind == "tiny":
        return q * 1e-260
    if kind == "huge":
        return q * 1e140
    if kind == "spread":    # neighbouring cells 12 decades apart
        return q * 10.0 ** rng.uniform(-12, 0, len(pos))
    return q


@pytest.mark.parametrize("n,p,depth", [(1, 4, 2), (9, 2, 3), (129, 3, 2), (600, 16, 3),
                                       (3000, 8, 4), (6000, 12, 3)])
@pytest.mark.parametrize("kind", ["plain", "zeros", "tiny", "huge", "spread"])
def test_fp64_default_equals_the_cuda_core_schedules(n, p, depth, kind):
    pos = W.sphere_sweep(max(n, 2), seed=9)["pos"][:n]
    q = charges(kind, pos)
    E, phi = far(pos, q, p, depth, "fp64")
    for schedule in ("tiles", "pairs"):
        Es, phis = far(pos, q, p, depth, "fp64", schedule)
        if not np.any(Es):
            assert not np.any(E)
            continue
        assert rel(E, Es) < 1e-12 and rel(phi, phis) < 1e-12, schedule


def test_fp64_nan_charge_stays_with_its_targets():
    pos = W.sphere_sweep(3000, seed=9)["pos"]
    q = charges("plain", pos)
    q[17] = np.nan
    E, _ = far(pos, q, 6, 4, "fp64")
    Es, _ = far(pos, q, 6, 4, "fp64", "tiles")
    assert np.array_equal(np.isnan(E), np.isnan(Es)) and np.isnan(E).any()
    ok = ~np.isnan(E)
    assert ok.any() and rel(E[ok], Es[ok]) < 1e-12


@pytest.mark.parametrize("p,depth", [(3, -1), (2, 6)])
def test_fp64_batches_equal_the_tile_schedule(p, depth):
    # beyond 262,144 ions: several batches of targets, a pool each
    pos = W.sphere_sweep(270001, seed=6)["pos"]
    q = charges("plain", pos)
    E, phi = far(pos, q, p, depth, "fp64")
    Es, phis = far(pos, q, p, depth, "fp64", "tiles")
    assert rel(E, Es) < 1e-12 and rel(phi, phis) < 1e-12


def test_fp64_plan_without_memory_for_its_digits_runs_on_the_cuda_cores():
    n, p = 270001, 4
    pos = W.sphere_sweep(n, seed=6)["pos"]
    q = charges("plain", pos)
    Es, _ = far(pos, q, p, -1, "fp64", "tiles")
    need = sum(pt.plan_footprint(n, p, precision="fp64"))
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - need + (400 << 20), dtype=torch.uint8, device=DEV)
    try:
        E, _ = far(pos, q, p, -1, "fp64")
    finally:
        del hog
        torch.cuda.empty_cache()
    assert rel(E, Es) < 1e-12


@pytest.mark.parametrize("n,p,depth", [(9, 2, 3), (65, 3, 2), (600, 5, 3), (3000, 8, 4),
                                       (6000, 12, 3), (5000, 13, 3), (4000, 16, 3)])
@pytest.mark.parametrize("schedule", ["tiles", "pairs"])
def test_fp32_schedules_match_fp64(n, p, depth, schedule):
    pos = W.sphere_sweep(n, seed=9)["pos"]
    q = charges("plain", pos)
    E, phi = far(pos, q, p, depth, "fp32", schedule)
    Ed, phid = far(pos, q, p, depth, "fp64", "tiles")
    if not np.any(Ed):
        assert not np.any(E)
        return
    assert rel(E, Ed) < 4e-6 and rel(phi, phid) < 4e-6
