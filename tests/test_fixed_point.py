"""The 64-bit fixed-point sines, cosines and angles behind the FP64-function sweeps and the FP64
energies: the header's integer code on the CPU against extended precision, and the kernels that use
it against the oracle where they can go wrong (edges of tiles and strips, angles outside the fixed
range, small local fields).
"""
import math
import os
import subprocess

import numpy as np
import pytest

import mpr_inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1910_08448_gb300", "csrc")
LD = np.longdouble
TWO_PI_LD = LD("6.283185307179586476925286766559005768")

HARNESS = r"""
#include <stdio.h>
#include "mpr_fixed.cuh"
using namespace mpr::fixed;
static constexpr DirTable T = make_dirs();
int main()
{
    char m;
    unsigned long long t;
    long long hx, hy;
    double x, q;
    int t0;
    while (scanf(" %c", &m) == 1) {
        if (m == 's' && scanf("%llu", &t) == 1) {
            int64_t c, s;
            sincos_turn(T.d, t, &c, &s);
            printf("%lld %lld\n", (long long)c, (long long)s);
        } else if (m == 't' && scanf("%la %la", &x, &q) == 2) {
            printf("%llu %llu\n", (unsigned long long)turns(x, split(turn_factor(q))),
                   (unsigned long long)turns((float)x, split(turn_factor(q))));
        } else if (m == 'a' && scanf("%lld %lld %d", &hx, &hy, &t0) == 3) {
            printf("%llu\n", (unsigned long long)doubled_arg(T.d, hx, hy, t0));
        } else if (m == 'd' && scanf("%llu", &t) == 1) {
            printf("%a\n", to_double_q60(t));
        }
    }
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(lines):
        r = subprocess.run([str(exe)], input="\n".join(lines) + "\n", capture_output=True,
                           text=True, check=True)
        return [ln.split() for ln in r.stdout.strip().split("\n")]

    return run


def _turn_rad(t):
    return TWO_PI_LD * LD(int(t) >> 32) / LD(2) ** 32 + TWO_PI_LD * LD(int(t) & 0xFFFFFFFF) / LD(2) ** 64


def _turn_gap(t, want):
    """Distance on the circle, in radians, of the turn t from `want` (in turns, extended)."""
    d = LD(int(t) >> 32) / LD(2) ** 32 - want + LD(int(t) & 0xFFFFFFFF) / LD(2) ** 64
    return abs(d - np.rint(d)) * TWO_PI_LD


def test_sine_and_cosine(harness):
    rng = np.random.default_rng(1)
    edges = [(k << 54) + (1 << 53) + e for k in range(0, 1024, 31) for e in (-1, 0, 1)]
    ts = [0, 1, 2**64 - 1, 2**62, 2**63, 2**61] + edges + [
        int(a) << 32 | int(b) for a, b in rng.integers(0, 2**32, size=(4000, 2))]
    ts = [t % 2**64 for t in ts]
    worst = 0.0
    for t, (c, s) in zip(ts, harness([f"s {t}" for t in ts])):
        a = _turn_rad(t)
        worst = max(worst, abs(LD(int(c)) / LD(2) ** 62 - np.cos(a)),
                    abs(LD(int(s)) / LD(2) ** 62 - np.sin(a)))
    # six truncated products of the series and the rotation: below 2^-58 each of the two largest
    assert worst <= 2.0**-57


def test_turns_of_an_angle(harness):
    rng = np.random.default_rng(2)
    xq = [(0.0, 0.5), (5e-324, 1.0), (7.499999999999999, 1.0), (2 * math.pi, 0.5), (2 * math.pi, 1.0),
          (2.0**-30, 0.5)]
    xq += [(float(x), float(q)) for x, q in zip(rng.uniform(0, 7.5, 2000), rng.uniform(1e-6, 1, 2000))]
    for (x, q), (td, tf) in zip(xq, harness([f"t {x.hex()} {q.hex()}" for x, q in xq])):
        assert _turn_gap(td, LD(x) * LD(q) / TWO_PI_LD) <= 2.0**-56.5
        if np.float32(x) < 7.5:
            assert _turn_gap(tf, LD(np.float32(x)) * LD(q) / TWO_PI_LD) <= 2.0**-56.5


def test_doubled_argument(harness):
    rng = np.random.default_rng(3)
    rows = []
    for r in (4.0, 1.0, 0.1, 2.0**-9):
        for a in list(rng.uniform(-math.pi, math.pi, 300)) + [0.0, math.pi / 2, -math.pi / 2, math.pi]:
            hx, hy = int(r * math.cos(a) * 2.0**60), int(r * math.sin(a) * 2.0**60)
            eps = rng.uniform(-1, 1) * (2e-7 if r > 0.01 else 4e-6)
            half = math.remainder(2 * (math.atan2(hy, hx) + eps), 2 * math.pi) / 2
            rows.append((hx, hy, round(half / (2 * math.pi) * 2**32), r))
    got = harness([f"a {hx} {hy} {t0}" for hx, hy, t0, _ in rows])
    for (hx, hy, _, r), (t,) in zip(rows, got):
        want = np.arctan2(LD(hy), LD(hx)) / TWO_PI_LD * 2
        # products with 58 bits over |h|, and the quotient's 2^-45 of a rest below 2^-18
        assert _turn_gap(t, want) <= 2.0**-55.5 / min(r, 1.0) + 2.0**-58, (hx, hy)


def test_rounding_to_fp64(harness):
    rng = np.random.default_rng(4)
    vs = [0, 1, 2**53 + 1, 2**54 + 2, 2**54 + 6, 2**62 - 1, 2**63 - 1]
    vs += [int(v) >> int(s) for v, s in zip(rng.integers(0, 2**63, 2000), rng.integers(0, 62, 2000))]
    for v, (d,) in zip(vs, harness([f"d {v}" for v in vs])):
        assert float.fromhex(d) == v / 2**60   # Python rounds the quotient of two integers once


# --- on the GPU -----------------------------------------------------------------------------------

@pytest.fixture(scope="module")
def mpr():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1910_08448_gb300 as m

    m.load()
    return m


def _half_sweeps(mpr, pr, setup, q, state, T, sweep, width=0.0):
    h = mpr.mpr_create(pr.z, pr.mask)
    try:
        mpr.mpr_set_options(h, setup, seed=11, q=q)
        mpr.mpr_set_state(h, state, sweep)
        mpr.mpr_set_temperature(h, T)
        if width:
            mpr.mpr_set_proposal(h, width)
        mpr.mpr_run(h, 1, 0)
        return mpr.mpr_get_state(h)[0]
    finally:
        mpr.mpr_destroy(h)


def _compare(orc, pr, q, state, T, sweep, got, tol=1e-9):
    o = orc.Oracle(pr.Lx, pr.Ly, seed=11, ubits=32, q=q)
    exp, mm, om = o.sweep(state, pr.mask, T, sweep, margins=True)
    col = (np.arange(pr.Ly)[:, None] + np.arange(pr.Lx)[None, :]) % 2
    bad = (mm < 1e-11) | (om < 1e-11)
    nb = np.zeros_like(bad)
    rb = bad & (col == 0)
    nb[:, 1:] |= rb[:, :-1]
    nb[:, :-1] |= rb[:, 1:]
    nb[1:] |= rb[:-1]
    nb[:-1] |= rb[1:]
    ok = ~(bad | (nb & (col == 1)))
    assert ok.mean() > 0.99
    assert np.abs(got - exp)[ok].max() <= tol


@pytest.mark.gpu
@pytest.mark.parametrize("Lx,Ly", [(2, 17), (126, 15), (128, 16), (130, 17), (257, 33)])
@pytest.mark.parametrize("far", [False, True])
def test_fp64_sweep_tile_edges(mpr, orc, Lx, Ly, far):
    """Edges of the 64 x 16 tiles; `far`: prediction angles outside [0, 7.5) in some tiles only."""
    pr = mpr_inputs.make_problem(Lx, Ly, 0.6, field_seed=21, mask_seed=22)
    o = orc.Oracle(Lx, Ly, seed=11, ubits=32)
    phi, _, _ = o.map(pr.z, pr.mask)
    rng = np.random.default_rng(5)
    state = np.where(pr.mask == 1, phi, rng.random((Ly, Lx)) * 2 * math.pi)
    if far:
        free = np.argwhere(pr.mask == 0)
        for y, x in free[:: max(1, len(free) // 3)]:
            state[y, x] = rng.choice([-0.5, 7.6, 11.0, -6.0])
    got = _half_sweeps(mpr, pr, "DDD", 0.5, state, 0.2, 6)
    _compare(orc, pr, 0.5, state, 0.2, 6, got)


@pytest.mark.gpu
@pytest.mark.parametrize("T", [1e-3, 10.0, 1e6])
def test_fp64_sweep_temperatures(mpr, orc, T):
    """The FP32 estimates of the acceptance test at the ends of the tuning's range and beyond."""
    pr = mpr_inputs.make_problem(200, 90, 0.9, field_seed=23, mask_seed=24)
    o = orc.Oracle(200, 90, seed=11, ubits=32)
    phi, _, _ = o.map(pr.z, pr.mask)
    rng = np.random.default_rng(6)
    state = np.where(pr.mask == 1, phi, rng.random((90, 200)) * 2 * math.pi)
    _compare(orc, pr, 0.5, state, T, 6, _half_sweeps(mpr, pr, "DDD", 0.5, state, T, 6))


@pytest.mark.gpu
def test_fp64_sweep_small_fields(mpr, orc):
    """q = 1 and neighbours in nearly opposite pairs: local fields from 1e-2 down to 1e-6, on both
    sides of the bound below which the FP64 functions take over."""
    Lx, Ly = 64, 48
    pr = mpr_inputs.make_problem(Lx, Ly, 0.5, field_seed=25, mask_seed=26)
    o = orc.Oracle(Lx, Ly, seed=11, ubits=32, q=1.0)
    phi, _, _ = o.map(pr.z, pr.mask)
    yy, xx = np.meshgrid(np.arange(Ly), np.arange(Lx), indexing="ij")
    rng = np.random.default_rng(7)
    eps = 10.0 ** rng.uniform(-6, -2, size=(Ly, Lx))
    # columns alternate by a half turn every two sites: left and right (up and down) neighbours of
    # a site are opposite up to eps
    base = 1.0 + math.pi * (((xx // 2) + (yy // 2)) % 2) + eps
    state = np.where(pr.mask == 1, phi, base)
    got = _half_sweeps(mpr, pr, "DDD", 1.0, state, 0.5, 6)
    # the red half alone: black sites see red results whose angles are off by 1e-16 / |h|
    exp, mm, om = o.half_sweep(state, pr.mask, 0.5, 6, 0)
    sel = ((xx + yy) % 2 == 0) & (mm >= 1e-9) & (om >= 1e-9)
    assert np.abs(got - exp)[sel].max() <= 1e-9   # 3e-16 / 1e-6, and the reflection doubles it


@pytest.mark.gpu
@pytest.mark.parametrize("Lx,Ly", [(2, 2), (30, 3), (31, 2), (32, 17), (61, 16), (63, 40), (700, 333)])
@pytest.mark.parametrize("q", [0.5, 1.0, 0.3])
@pytest.mark.parametrize("far", [False, True])
def test_energies(mpr, Lx, Ly, q, far):
    """Both energies at the edges of their strips; `far`: some angles outside the fixed range."""
    import torch

    rng = np.random.default_rng(8)
    phi = rng.random((Ly, Lx)) * 2 * math.pi
    if far:
        for _ in range(3):
            phi[rng.integers(Ly), rng.integers(Lx)] = rng.choice([-3.0, 9.0, -20.0, 7.5])
    a = phi.astype(LD)
    total = np.cos(LD(q) * (a[:, 1:] - a[:, :-1])).sum() + np.cos(LD(q) * (a[1:] - a[:-1])).sum()
    want = float(-total / (Lx * (Ly - 1) + Ly * (Lx - 1)))
    t = torch.from_numpy(phi).cuda()
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    mpr.mpr_bond_energy_noalloc(t, q, out)
    tol = 4e-16   # terms to 2^-51, a mean of at most 1 rounded a few times
    assert abs(float(out.cpu()[0]) - want) <= tol + (1e-15 if far else 0.0)
    mask = np.zeros((Ly, Lx), dtype=np.uint8)
    mask[0, :2] = 1
    z = np.where(mask == 1, np.arange(Lx)[None, :], 0.0) + np.zeros((Ly, Lx))
    h = mpr.mpr_create(z, mask)
    try:
        mpr.mpr_set_options(h, "DDS", q=q)
        mpr.mpr_set_state(h, phi, 0)
        b, _ = mpr.mpr_get_state(h)
        b = b.astype(LD)
        total = np.cos(LD(q) * (b[:, 1:] - b[:, :-1])).sum() + np.cos(LD(q) * (b[1:] - b[:-1])).sum()
        want = float(-total / (Lx * (Ly - 1) + Ly * (Lx - 1)))
        assert abs(mpr.mpr_energy(h)[0] - want) <= tol + (1e-15 if far else 0.0)
    finally:
        mpr.mpr_destroy(h)


@pytest.mark.gpu
def test_energy_of_not_a_number(mpr):
    import torch

    phi = torch.full((40, 50), 1.0, dtype=torch.float64, device="cuda")
    phi[7, 9] = math.nan
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    mpr.mpr_bond_energy_noalloc(phi, 0.5, out)
    assert math.isnan(float(out.cpu()[0]))
