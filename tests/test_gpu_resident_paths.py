"""The resident sweep kernel is the one that runs where it should: one launch for a plain run, three for a
measured one (the sweeps, their tile partials, the sums), against two a sweep of the tile kernel;
alone and with another thread's handle in between.
"""
import threading

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


def _launches(mpr, h, equil, samples):
    before = mpr.mpr_get_info(h)["kernel_launches"]
    mpr.mpr_run(h, equil, samples)
    return mpr.mpr_get_info(h)["kernel_launches"] - before


def _handle(mpr, pr, setup="SDS", kind=-1, stream=None):
    h = mpr.mpr_create(pr.z, pr.mask)
    if stream is not None:
        mpr.mpr_set_stream(h, stream)
    mpr.mpr_set_options(h, setup, seed=31)
    mpr.mpr_set_sweep_kernel(h, kind)
    mpr.mpr_set_temperature(h, 0.2)
    return h


def _problem(Lx, Ly, seed=61):
    pr = mpr_inputs.make_problem(Lx, Ly, 0.6, field_seed=seed, mask_seed=seed + 1, periodic=True)
    pr.mask[0, :2] = 1
    return pr


# a cluster that exchanges rows every 4 or 2 passes, a grid every 4 or 2, every pass with rows and with row
# pairs; a single band; the widest and the tallest
@pytest.mark.parametrize("Lx,Ly", [(40, 64), (64, 63), (9, 200), (112, 97), (128, 127), (60, 400), (61, 399),
                                   (90, 767), (250, 100), (256, 255), (301, 299), (400, 300), (512, 401),
                                   (2, 2500), (1200, 3), (1400, 1200), (777, 523), (1024, 1024)])
@pytest.mark.parametrize("setup", ["SDS", "HDS"])
def test_the_resident_kernel_runs(mpr, Lx, Ly, setup):
    h = _handle(mpr, _problem(Lx, Ly), setup)
    try:
        assert _launches(mpr, h, 4, 0) == 1
        assert _launches(mpr, h, 37, 0) == 1
        assert _launches(mpr, h, 0, 3) == 3
        mpr.mpr_set_sweep_kernel(h, 0)
        assert _launches(mpr, h, 5, 0) == 10
    finally:
        mpr.mpr_destroy(h)


@pytest.mark.parametrize("shapes", [((1024, 1024), (900, 900)), ((777, 523), (700, 400))])
def test_two_sizes_on_two_threads(mpr, shapes):
    """Short runs of two lattices of one resident kernel, of different shared memory."""
    import torch

    n, prs = 60, [_problem(*s, seed=71 + i) for i, s in enumerate(shapes)]

    def work(i, kind, stream, out):
        h = _handle(mpr, prs[i], kind=kind, stream=stream)
        try:
            launches = sum(_launches(mpr, h, 2, 0) + _launches(mpr, h, 0, 2) for _ in range(n))
            out[i] = (mpr.mpr_get_state(h)[0], mpr.mpr_predict(h), launches)
        finally:
            mpr.mpr_destroy(h)

    want, got = [None, None], [None, None]
    for i in range(2):
        work(i, 0, None, want)
    ts = [threading.Thread(target=work, args=(i, -1, torch.cuda.Stream(), got)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for g, w in zip(got, want):
        assert np.array_equal(g[0], w[0]) and np.array_equal(g[1], w[1])
        assert g[2] == n * (1 + 3) and w[2] == n * (4 + 5)


# one sweep behind a resident launch, which runs the tile kernel: on a cluster, a grid every 4 and 2 passes,
# rows and row pairs
@pytest.mark.parametrize("Lx,Ly", [(64, 64), (128, 127), (90, 767), (400, 300), (777, 523), (1400, 1200)])
@pytest.mark.parametrize("setup", ["SDS", "HDS", "BSS"])
def test_one_sweep_behind_a_resident_launch(mpr, Lx, Ly, setup):
    pr, out = _problem(Lx, Ly), []
    for kind in (-1, 0):
        h = _handle(mpr, pr, setup, kind)
        try:
            for equil in (4, 25, 5, 4097, 7):
                mpr.mpr_run(h, equil, 1)
            out.append((mpr.mpr_get_state(h)[0], mpr.mpr_predict(h), mpr.mpr_get_info(h)["e_bond_mean"]))
        finally:
            mpr.mpr_destroy(h)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]


# the shortest resident runs, two and three sweeps, on a cluster that exchanges rows every 4 passes and every 2, on
# both grids, rows and row pairs
@pytest.mark.parametrize("Lx,Ly", [(66, 64), (128, 127), (90, 767), (300, 300), (512, 401), (1400, 1200), (12, 60000)])
@pytest.mark.parametrize("setup", ["SDS", "HDS"])
def test_the_shortest_resident_runs(mpr, Lx, Ly, setup):
    pr, out = _problem(Lx, Ly), []
    for kind in (-1, 0):
        h = _handle(mpr, pr, setup, kind)
        try:
            n = [_launches(mpr, h, *call) for call in ((2, 0), (3, 0), (0, 2), (0, 3))]
            assert n == ([1, 1, 3, 3] if kind else [4, 6, 5, 7])
            out.append((mpr.mpr_get_state(h)[0], mpr.mpr_predict(h), mpr.mpr_get_info(h)["e_bond_mean"]))
        finally:
            mpr.mpr_destroy(h)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]


# the first band withholds its rows: its neighbour's bounded wait runs out, every block leaves, the error is
# reported once and the handle goes on (fine grid of 17 and of 150 bands, one row and row pairs per thread)
@pytest.mark.parametrize("Lx,Ly", [(258, 34), (300, 300), (777, 523), (1024, 1024)])
@pytest.mark.parametrize("call", [(40, 0), (7, 20)])
def test_a_wait_that_runs_out_is_reported(mpr, Lx, Ly, call):
    pr = _problem(Lx, Ly)
    h = _handle(mpr, pr)
    try:
        want = []
        for stall in (True, False):
            mpr.mpr_set_options(h, "SDS", seed=31)
            mpr.mpr_set_temperature(h, 0.2)
            mpr.mpr_run(h, 4, 0)
            if stall:
                mpr.mpr_inject_tma_stall(h, 0.05)
                with pytest.raises(mpr.MPRError) as e:
                    mpr.mpr_run(h, *call)
                assert e.value.status == mpr.MPR_ERR_DEVICE_TIMEOUT
                state, sweep = mpr.mpr_get_state(h)
                assert sweep == 4 + sum(call) and state.min() >= 0.0 and state.max() <= 6.2831855
                mpr.mpr_set_options(h, "SDS", seed=31)
                mpr.mpr_set_temperature(h, 0.2)
                mpr.mpr_run(h, 4, 0)
            mpr.mpr_run(h, 30, 20)   # tags of the run that was cut off are never taken for new ones
            want.append((mpr.mpr_get_state(h)[0], mpr.mpr_predict(h), mpr.mpr_get_info(h)["e_bond_mean"]))
        assert np.array_equal(want[0][0], want[1][0]) and np.array_equal(want[0][1], want[1][1])
        assert want[0][2] == want[1][2]
    finally:
        mpr.mpr_destroy(h)
