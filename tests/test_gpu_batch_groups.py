"""Graph mode runs groups of problems side by side, some sweeps per turn of each loop: the results are
the bits of the persistent kernel, which runs all problems as one group sweep by sweep.
"""
import numpy as np
import pytest

import mpr_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mpr():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1910_08448_gb300 as m

    m.load()
    return m


def _fills(mpr, prs, setup, mode, calls):
    b = mpr.mpr_batch_create([p.z for p in prs], [p.mask for p in prs], setup, seed=5)
    try:
        mpr.mpr_batch_set_tuning(b, n_eq=20, n_meas=10)
        mpr.mpr_batch_set_launch(b, mode=mode)
        out = []
        for equil, samples, T in calls:
            t, st = mpr.mpr_batch_fill(b, equil, samples, None if T is None else [T] * len(prs))
            out += [t, st, mpr.mpr_batch_get_stats(b)["iterations"]]
            for i in range(len(prs)):
                state, sweep = mpr.mpr_batch_get_state(b, i)
                info = mpr.mpr_batch_get_info(b, i)
                out += [state, sweep, info["e_bond_mean"], info["site_updates"]]
                if info["n_samples"]:
                    out.append(mpr.mpr_batch_predict(b, i))
        return out
    finally:
        mpr.mpr_batch_destroy(b)


# fewer problems than groups, as many, more (with equal and uneven sizes); runs of fewer sweeps than a
# turn, of a turn, of one more
@pytest.mark.parametrize("n", [1, 7, 8, 21])
@pytest.mark.parametrize("setup", ["SDS", "HDS"])
def test_groups_give_the_bits_of_one_group(mpr, n, setup):
    prs = []
    for i in range(n):
        Lx, Ly = (33 + 41 * (i * i % 11), 20 + 37 * (i * 5 % 7)) if i else (300, 40)
        pr = mpr_inputs.make_problem(Lx, Ly, (0.33, 0.66, 0.9)[i % 3], field_seed=70 + i, mask_seed=90 + i,
                                     periodic=True)
        pr.mask[0, :2] = 1
        prs.append(pr)
    calls = [(1, 0, 0.2), (3, 5, 0.2), (8, 1, 0.3), (12, 20, None), (0, 17, 0.1)]
    for g, w in zip(_fills(mpr, prs, setup, 2, calls), _fills(mpr, prs, setup, 0, calls)):
        assert np.array_equal(g, w, equal_nan=True)
