"""Plain passes of the tile kernel that run some or all of their tiles as half-height tiles: the states
are the bits of measured passes, whose black passes always run whole tiles.
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


def _state(mpr, pr, setup, bounded, equil, samples, q):
    h = mpr.mpr_create(pr.z, pr.mask)
    try:
        mpr.mpr_set_options(h, setup, seed=11, q=q)
        mpr.mpr_set_sweep_kernel(h, 0)
        if bounded:
            mpr.mpr_set_proposal(h, 2.5, 0.0)
        mpr.mpr_set_temperature(h, 0.2)
        mpr.mpr_run(h, equil, samples)
        return mpr.mpr_get_state(h)[0]
    finally:
        mpr.mpr_destroy(h)


# last tile columns of 1, 32, 33, 64, 65 and 128 half-columns, heights around half and whole tiles;
# one wave; a last wave of few and of many tiles
SHAPES = [(2, 2), (258, 15), (320, 16), (322, 17), (384, 31), (386, 33), (512, 49), (777, 523), (2501, 1333),
          (2048, 2048), (2560, 2560), (3001, 3000)]


@pytest.mark.parametrize("Lx,Ly", SHAPES)
@pytest.mark.parametrize("setup,bounded,q", [("SDS", False, 0.5), ("HDS", False, 0.5), ("BDS", False, 0.8),
                                             ("HDH", False, 0.5), ("DDS", False, 0.5), ("SDS", True, 0.5),
                                             ("HDS", True, 0.5)])
def test_half_height_tiles_give_the_same_states(mpr, Lx, Ly, setup, bounded, q):
    pr = mpr_inputs.make_problem(Lx, Ly, 0.6, field_seed=21, mask_seed=22, periodic=True)
    pr.mask[0, :2] = 1
    assert np.array_equal(_state(mpr, pr, setup, bounded, 5, 0, q), _state(mpr, pr, setup, bounded, 0, 5, q))


@pytest.mark.parametrize("setup", ["HDS", "HSS"])
def test_energies_of_more_sweeps_than_one_sum_takes(mpr, setup):
    """8192^2: the partials of 64 (FP32 energies: 128) measured sweeps are summed at once."""
    pr = mpr_inputs.make_problem(8192, 8192, 0.9, field_seed=23, mask_seed=24, periodic=True)
    n = 64 if setup == "HDS" else 128
    means = []
    for runs in ((n + 5,), (n - 1, 6)):
        h = mpr.mpr_create(pr.z, pr.mask)
        try:
            mpr.mpr_set_options(h, setup, seed=3)
            mpr.mpr_set_temperature(h, 0.065)
            total = 0.0
            for r in runs:
                mpr.mpr_run(h, 0, r)
                total += r * mpr.mpr_get_info(h)["e_bond_mean"]
            means.append(total / (n + 5))
        finally:
            mpr.mpr_destroy(h)
    assert abs(means[0] - means[1]) <= 1e-13 * abs(means[1])
