"""The FP64 energies of small states, to the rounding of the result: the sum is exact but for its terms.

e_b = -S / N_b is rounded twice, S (at most N_b) to FP64 and the quotient (at most 1): each at most 2^-54 of e_b's
scale, rms 2^-54 / sqrt(3). The terms of S are good to 2^-55, their rms error is 2^-58.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble
MOST = 2.0**-53 + 2.0**-55
RMS = 2.0**-54 * math.sqrt(2.0 / 3.0) + 2.0**-57


@pytest.fixture(scope="module")
def mpr():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1910_08448_gb300 as m

    m.load()
    return m


def _exact(phi, q):
    """e_b of a stack of states in extended precision."""
    a = phi.astype(LD) * LD(q)
    Ly, Lx = phi.shape[-2:]
    s = np.cos(a[..., 1:] - a[..., :-1]).sum((-1, -2)) + np.cos(a[..., 1:, :] - a[..., :-1, :]).sum((-1, -2))
    return -s / LD(Lx * (Ly - 1) + Ly * (Lx - 1))


def _within(err):
    assert np.abs(err).max() <= MOST
    assert math.sqrt(float((err.astype(np.float64) ** 2).mean())) <= RMS


@pytest.mark.parametrize("Lx,Ly", [(2, 2), (3, 2), (2, 5), (4, 4), (8, 8), (33, 17), (200, 150)])
@pytest.mark.parametrize("q", [0.5, 1.0, 0.3])
def test_state_energies_are_rounded_twice(mpr, Lx, Ly, q):
    import torch

    n = 2000 if Lx * Ly <= 64 else 100
    phi = np.random.default_rng(41).random((n, Ly, Lx)) * 2 * math.pi
    t, out = torch.from_numpy(phi).cuda(), torch.zeros(n, dtype=torch.float64, device="cuda")
    for i in range(n):
        mpr.mpr_bond_energy_noalloc(t[i], q, out[i : i + 1])
    _within(out.cpu().numpy().astype(LD) - _exact(phi, q))
    mask = np.zeros((Ly, Lx), dtype=np.uint8)
    mask[0, :2] = 1
    h = mpr.mpr_create(np.arange(Lx)[None, :] + np.zeros((Ly, Lx)), mask)
    try:
        mpr.mpr_set_options(h, "DDD", q=q)
        e, states = [], []
        for i in range(min(n, 400)):
            mpr.mpr_set_state(h, phi[i], 0)
            states.append(mpr.mpr_get_state(h)[0])
            e.append(mpr.mpr_energy(h)[0])
        _within(np.array(e).astype(LD) - _exact(np.array(states), q))
    finally:
        mpr.mpr_destroy(h)


# a few columns, where a warp walks several strips side by side: widths around each strip width, last strips of
# every height, angles outside the fixed range in some strips
@pytest.mark.parametrize("Lx", [2, 3, 4, 5, 11, 12, 13, 27, 28, 29])
@pytest.mark.parametrize("Ly", [2, 7, 33, 30011])
@pytest.mark.parametrize("setup,far", [("DDD", False), ("HDS", False), ("DDD", True)])
def test_state_energies_of_narrow_grids(mpr, Lx, Ly, setup, far):
    rng = np.random.default_rng(42)
    phi = rng.random((Ly, Lx)) * 2 * math.pi
    if far:
        for _ in range(3):
            phi[rng.integers(1, Ly), rng.integers(Lx)] = rng.choice([-3.0, 9.0, 7.5])
    mask = np.zeros((Ly, Lx), dtype=np.uint8)
    mask[0, :2] = 1
    h = mpr.mpr_create(np.arange(Lx)[None, :] + np.zeros((Ly, Lx)), mask)
    try:
        mpr.mpr_set_options(h, setup)
        mpr.mpr_set_state(h, phi, 0)
        err = LD(mpr.mpr_energy(h)[0]) - _exact(mpr.mpr_get_state(h)[0], 0.5)
    finally:
        mpr.mpr_destroy(h)
    # out of range: five FP64 sincos and products per site, below 2^-50 each
    assert abs(err) <= MOST + (2.0**-50 if far else 0.0)
