"""The map from mean angles back to data, zmin + (zmax - zmin) * mean / (2 pi): over data ranges down to the
smallest FP64 numbers, and on grids of any shape.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble
TWO_PI_LD = LD("6.283185307179586476925286766559005768")


@pytest.fixture(scope="module")
def mpr():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1910_08448_gb300 as m

    m.load()
    return m


def _check(mpr, z, mask, setup, acc, n):
    """The prediction from n samples, each taken by a sweep whose angles are read back."""
    Ly, Lx = z.shape
    h = mpr.mpr_create(z, mask)
    try:
        mpr.mpr_set_options(h, setup, seed=5, acc=acc)
        mpr.mpr_set_temperature(h, 0.3)
        total = np.zeros((Ly, Lx), dtype=LD)
        for _ in range(n):
            mpr.mpr_run(h, 0, 1)
            total += mpr.mpr_get_state(h)[0].astype(LD)
        got = mpr.mpr_predict(h)
    finally:
        mpr.mpr_destroy(h)
    lo, hi = z[mask != 0].min(), z[mask != 0].max()
    want = LD(lo) + (LD(hi) - LD(lo)) * (total / n / TWO_PI_LD)
    free = mask == 0
    assert np.array_equal(got[~free], z[~free])
    # zmax - zmin, 2 pi n, their quotient and the result are rounded (2^-53 each); n sums in FP64, or
    # compensated in FP32 (2^-22.9 of the sum: two roundings of the last terms)
    scale = float(hi - lo)
    tol = scale * (2.0**-51 + n * 2.0**-52 if acc == "f64" else 2.0**-22) + max(abs(lo), abs(hi)) * 2.0**-52
    assert np.abs((got - want)[free].astype(np.float64)).max(initial=0.0) <= max(tol, 5e-324)


@pytest.mark.parametrize("unit", [1.0, 1e-300, 3e-307, 1e-310, 5e-324, 1e300])
@pytest.mark.parametrize("setup,acc", [("DDD", "f64"), ("SDS", "f64"), ("HDS", "kahan")])
def test_any_range(mpr, unit, setup, acc):
    rng = np.random.default_rng(1)
    z = np.rint(rng.uniform(1, 100, (40, 33))) * unit
    mask = (rng.random((40, 33)) < 0.4).astype(np.uint8)
    mask[0, :2] = 1
    _check(mpr, z, mask, setup, acc, 3)


# widths around the powers of two that a block's columns are rounded to; heights around its rows
@pytest.mark.parametrize("Lx", [2, 3, 4, 5, 31, 33, 64, 65, 128, 129, 257])
@pytest.mark.parametrize("Ly", [2, 9, 1030])
def test_any_shape(mpr, Lx, Ly):
    rng = np.random.default_rng(2)
    z, mask = rng.normal(50, 10, (Ly, Lx)), (rng.random((Ly, Lx)) < 0.4).astype(np.uint8)
    mask[0, :2] = 1
    _check(mpr, z, mask, "SDS", "f64", 2)


# grids of many blocks, where a thread takes several rows (the sizes above take one): last blocks of few rows
@pytest.mark.parametrize("Lx,Ly", [(2, 400007), (5, 100003), (64, 12001), (129, 2500), (257, 2003), (2003, 400)])
@pytest.mark.parametrize("acc", ["f64", "kahan"])
def test_several_rows_per_thread(mpr, Lx, Ly, acc):
    rng = np.random.default_rng(3)
    z, mask = rng.normal(50, 10, (Ly, Lx)), (rng.random((Ly, Lx)) < 0.4).astype(np.uint8)
    _check(mpr, z, mask, "SDS", acc, 2)
