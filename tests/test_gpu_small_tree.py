"""The tree of up to 2,048 ions in one launch against the general tree's kernels.
"""
import numpy as np
import pytest

import paper_2405_13973_gb300 as pt
import workloads as W

pytestmark = pytest.mark.gpu


def rel(a, b):
    m = np.abs(b).max()
    return float(np.linalg.norm((a - b) / m) / np.linalg.norm(b / m))


@pytest.mark.parametrize("precision,depth", [("fp64", 0), ("fp64", 2), ("fp64", 4), ("bf16x3", 1),
                                             ("tf32x3", 3), ("fp32", 5)])
def test_steps_of_the_one_launch_tree_equal_the_general_tree(precision, depth):
    # ions of zero charge carry a crystal of 2,000 over the line at 2,048: the
    # charged ions' cells stay, so do their trajectories (1e-9 of the extent
    # in FP64 after 4 steps, the field's 4e-6 times the field's share of the
    # motion otherwise; a misplaced ion shows at 1e-3)
    cr = W.ensemble_member(2000, 0.5, seed=5)
    rng = np.random.default_rng(4)
    i = rng.permutation(2000)[:49]
    j = (i + 1 + rng.integers(0, 1999, 49)) % 2000
    extra = 0.5 * (cr["pos"][i] + cr["pos"][j])
    out = []
    for k in (47, 48, 49):
        pos = np.concatenate([cr["pos"], extra[:k]])
        vel = np.concatenate([cr["vel"], np.zeros((k, 3))])
        q = np.concatenate([cr["q"], np.zeros(k)])
        plan = pt.Plan(len(q), p=6, depth=depth, precision=precision)
        st = pt.State.from_numpy(pos, vel, q)
        plan.step(st, cr["trap"], pt.make_laser(cr["beams"], seed=3, gamma0=W.GAMMA0), cr["dt"], 4)
        out.append((st.pos().cpu().numpy()[:2000], st.vel().cpu().numpy()[:2000]))
        plan.close()
    tol = 1e-9 if precision == "fp64" else 4e-6
    for x, v in out[:2]:
        assert rel(x, out[2][0]) < tol and rel(v, out[2][1]) < tol
