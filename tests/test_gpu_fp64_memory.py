"""FP64 plans that cannot get the memory of the tensor-core translations run the
CUDA-core tiles, the same bits as a plan that was asked for them, and keep
none of what the others would have needed.  Both ways to run out: the plan's
digits and pool of partial rows (kept for more than 262,144 ions), and the
operators' digits, which are allocated last.
"""
import numpy as np
import pytest
import torch

import paper_2405_13973_gb300 as pt
import workloads as W

pytestmark = pytest.mark.gpu


def operator_digit_bytes(p):
    P = (p + 1) ** 2
    npad, k32 = (P + 15) // 16 * 16, (P + 31) // 32
    return 359 * (k32 * 7 * npad * 64 + npad * 2)


@pytest.mark.parametrize("short", ["pool", "operators"])
def test_without_memory_for_the_digits_the_tiles_run(short):
    n, p = 270001, 10
    w = W.sphere_sweep(n, seed=6)
    pos = torch.tensor(np.ascontiguousarray(w["pos"].T), device="cuda")
    q = torch.tensor(w["q"], device="cuda")

    def far(schedule=None):
        plan = pt.Plan(n, p=p, depth=5, precision="fp64")
        free = torch.cuda.mem_get_info()[0]
        if schedule:
            plan.set_m2l_schedule(schedule)
        plan.set_phases(pt.PT_PHASE_FAR)
        E, _ = plan.forces(pos, q)
        plan.close()
        return E, free

    tiles, default = far("tiles")[0], far()[0]
    assert not torch.equal(tiles, default)
    need = sum(pt.plan_footprint(n, p, depth=5, precision="fp64"))
    lack = operator_digit_bytes(p) // 2 if short == "operators" else 200 << 20
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - need + lack, dtype=torch.uint8, device="cuda")
    try:
        E, free = far()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert torch.equal(E, tiles)
    assert free > 256 << 20  # the pool is 512 MB at least, less what was lacking
