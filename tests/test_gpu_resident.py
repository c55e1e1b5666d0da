"""The resident sweep kernel (many sweeps in one launch, the lattice in shared memory) against the
one-launch-per-pass tile kernel: states, predictions and energies agree bit for bit, on lattices
of one band, of a cluster and of a grid of bands, with ragged last bands and columns, one row or a
row pair per thread, and several units per thread.
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


def _run(mpr, pr, setup, kind, T=0.2, q=0.5, acc="f64", parts=((7, 0), (0, 19), (14, 3)), stream=None):
    h = mpr.mpr_create(pr.z, pr.mask)
    try:
        if stream is not None:
            mpr.mpr_set_stream(h, stream)
        mpr.mpr_set_options(h, setup, seed=31, q=q, acc=acc)
        mpr.mpr_set_sweep_kernel(h, kind)
        mpr.mpr_set_temperature(h, T)
        e = []
        for equil, samples in parts:
            mpr.mpr_run(h, equil, samples)
            e.append(mpr.mpr_get_info(h)["e_bond_mean"])
        state, sweep = mpr.mpr_get_state(h)
        return state, sweep, mpr.mpr_predict(h), e, mpr.mpr_get_info(h)
    finally:
        mpr.mpr_destroy(h)


def _same(a, b):
    assert a[1] == b[1]
    assert np.array_equal(a[0], b[0])
    assert np.array_equal(a[2], b[2])
    assert a[3][1:] == b[3][1:]


SHAPES = [(2, 2), (2, 40), (5, 3), (64, 64), (63, 31), (128, 128), (131, 37), (129, 130), (257, 129),
          (300, 45), (777, 523), (1024, 1024), (1030, 611), (3000, 90), (90, 3000)]


@pytest.mark.parametrize("Lx,Ly", SHAPES)
@pytest.mark.parametrize("setup", ["SDS", "HDS"])
def test_same_bits_as_the_tile_kernel(mpr, Lx, Ly, setup):
    pr = mpr_inputs.make_problem(Lx, Ly, 0.6, field_seed=51, mask_seed=52, periodic=True)
    pr.mask[0, :2] = 1
    auto, tile = _run(mpr, pr, setup, -1), _run(mpr, pr, setup, 0)
    _same(auto, tile)
    assert auto[4]["sweep_kernel"] in (0, 1) and auto[4]["site_updates"] == tile[4]["site_updates"]


@pytest.mark.parametrize("setup,q,acc", [("SSS", 0.5, "kahan"), ("BDS", 0.7, "f64"), ("HSS", 1.0, "kahan"),
                                         ("SDS", 0.3, "f64"), ("BSS", 0.5, "f64"), ("DDS", 0.5, "f64"),
                                         ("HDH", 0.5, "f64")])
@pytest.mark.parametrize("Lx,Ly", [(101, 67), (300, 211)])
def test_same_bits_for_every_option(mpr, Lx, Ly, setup, q, acc):
    pr = mpr_inputs.make_problem(Lx, Ly, 0.6, field_seed=53, mask_seed=54)
    _same(_run(mpr, pr, setup, -1, q=q, acc=acc), _run(mpr, pr, setup, 0, q=q, acc=acc))


def test_many_sweeps_and_tuning(mpr):
    """A tuning and 400 sweeps: thousands of passes of tagged boundary rows."""
    for Lx, Ly in ((64, 64), (200, 150)):
        pr = mpr_inputs.make_problem(Lx, Ly, 0.33, field_seed=55, mask_seed=56)
        out = []
        for kind in (-1, 0):
            h = mpr.mpr_create(pr.z, pr.mask)
            try:
                mpr.mpr_set_sweep_kernel(h, kind)
                mpr.mpr_set_tuning(h, n_eq=40, n_meas=20)
                T, st = mpr.mpr_tune_temperature(h)
                mpr.mpr_run(h, 300, 100)
                out.append((T, st, mpr.mpr_get_state(h)[0], mpr.mpr_predict(h)))
            finally:
                mpr.mpr_destroy(h)
        assert out[0][:2] == out[1][:2]
        assert np.array_equal(out[0][2], out[1][2]) and np.array_equal(out[0][3], out[1][3])


def test_two_handles_on_two_streams(mpr):
    """Two host threads, a stream and a handle each, lattices whose bands fill the device."""
    import torch

    prs = [mpr_inputs.make_problem(512, 512, 0.6, field_seed=57 + i, mask_seed=58) for i in range(2)]
    want = [_run(mpr, pr, "SDS", 0, parts=((60, 0), (0, 20))) for pr in prs]
    got = [None, None]

    def work(i):
        s = torch.cuda.Stream()
        for _ in range(3):
            got[i] = _run(mpr, prs[i], "SDS", -1, parts=((60, 0), (0, 20)), stream=s)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for g, w in zip(got, want):
        _same(g, w)


# One plan of each kind at its edges: a cluster that exchanges rows every 4 or 2 passes, a grid every
# 4 or 2, or every pass with rows and with row pairs; odd heights whose last band is one row short;
# a single band; the widest and the tallest. Runs of 2 and 3 sweeps hold the fewest exchanges.
@pytest.mark.parametrize("Lx,Ly", [(40, 64), (64, 63), (9, 200), (112, 97), (128, 127), (60, 400), (61, 399),
                                   (90, 767), (250, 100), (256, 255), (301, 299), (400, 300), (512, 401),
                                   (2, 2500), (1200, 3), (1400, 1200)])
@pytest.mark.parametrize("setup,q,acc", [("SDS", 0.5, "f64"), ("HDS", 0.8, "kahan")])
def test_same_bits_for_every_plan(mpr, Lx, Ly, setup, q, acc):
    pr = mpr_inputs.make_problem(Lx, Ly, 0.6, field_seed=61, mask_seed=62, periodic=True)
    pr.mask[0, :2] = 1
    parts = ((2, 0), (3, 2), (0, 3), (1, 1), (25, 9))
    _same(_run(mpr, pr, setup, -1, q=q, acc=acc, parts=parts), _run(mpr, pr, setup, 0, q=q, acc=acc, parts=parts))


@pytest.mark.parametrize("Lx,Ly", [(64, 64), (300, 211), (700, 500)])
def test_more_sweeps_than_one_launch_takes(mpr, Lx, Ly):
    """4096 sweeps a launch: the remainder of one sweep joins the launch before it."""
    pr = mpr_inputs.make_problem(Lx, Ly, 0.6, field_seed=63, mask_seed=64, periodic=True)
    parts = ((4097, 0), (8193, 4))
    _same(_run(mpr, pr, "SDS", -1, parts=parts), _run(mpr, pr, "SDS", 0, parts=parts))
