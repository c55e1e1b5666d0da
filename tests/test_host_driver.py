"""The library's host code on a stand-in CUDA runtime, on the CPU: which launches a call makes, in which
order and with which attributes, and what it does when a launch or an allocation is refused.
"""
import glob
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.join(ROOT, "tests")


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    import __graft_entry__
    from paper_1910_08448_gb300 import _build

    __graft_entry__.build()
    objs = sorted(glob.glob(os.path.join(_build.BUILD, "mpr_*.o")))
    if len(objs) != len(_build.sources()):   # a library that was built elsewhere
        _build.build(force=True)
        objs = sorted(glob.glob(os.path.join(_build.BUILD, "mpr_*.o")))
    exe = str(tmp_path_factory.mktemp("driver") / "driver")
    cuda = os.path.join(os.path.dirname(os.path.dirname(_build.nvcc())), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", cuda, "-I", _build.INCLUDE, "-I", HERE,
                    os.path.join(HERE, "host_driver.cpp"), os.path.join(HERE, "fake_cudart.cpp"), *objs,
                    "-ldl", "-lpthread", "-o", exe], check=True)

    def run(*args):
        r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, (r.returncode, r.stderr)
        lines = r.stdout.strip().split("\n")
        out = []
        for ln in lines[1:]:
            name, *rest = ln.split()
            out.append((name, {k: int(v) for k, v in (p.split("=") for p in rest)}))
        return int(lines[0].split()[1]), out

    return run


def _resident(name):
    return "fine_kernel" in name or "coarse_kernel" in name


def _tile(name):
    return "sweep_f32_kernel" in name


# a larger lattice whose resident kernel is also the smaller one's (row pairs; one row; a grid of the
# fine kernel), and another handle's thread that runs in between
@pytest.mark.parametrize("big,small", [((1400, 1200), (1024, 1024)), ((777, 523), (700, 400)),
                                       ((300, 300), (200, 150))])
def test_a_smaller_lattice_leaves_the_shared_memory_of_a_larger_one(driver, big, small):
    status, calls = driver("other", *big, *small)
    assert status == 0
    names = [n for n, _ in calls]
    most = max(a["smem"] for n, a in calls if _resident(n))
    mine = [n for n, a in calls if _resident(n) and a["smem"] == most]
    assert len(mine) >= 2 and not any(_tile(n) for n in names)


REFUSED = {"cooperative launch too large": 720, "invalid cluster size": 912, "out of resources": 701}
OTHER = {"invalid value": 1, "invalid configuration": 9, "unknown": 999}


@pytest.mark.parametrize("shape", [(64, 64), (300, 300), (777, 523)])
def test_only_a_launch_that_is_too_large_falls_back(driver, shape):
    for code in REFUSED.values():
        status, calls = driver("refuse", *shape, code)
        assert status == 0 and sum(_tile(n) for n, _ in calls) == 2 * 9
    for code in OTHER.values():
        status, calls = driver("refuse", *shape, code)
        assert status == 5 and not any(_tile(n) for n, _ in calls)


# one sweep behind a resident launch: its first pass loads its own rows before it waits for the kernel in
# front, and the resident kernel wrote both colours
@pytest.mark.parametrize("shape", [(64, 64), (300, 300), (777, 523), (1400, 1200)])
def test_a_pass_behind_a_resident_launch_is_no_programmatic_dependent(driver, shape):
    for call in (("run", *shape, 4, 1), ("run", *shape, 25, 1), ("run", *shape, 4097, 1), ("tune", *shape, 5, 1)):
        status, calls = driver(*call)
        behind = [i for i in range(1, len(calls)) if _tile(calls[i][0]) and not _tile(calls[i - 1][0])]
        assert status in (0, 4) and behind and all(_resident(calls[i - 1][0]) for i in behind)
        for i in behind:
            assert calls[i][1]["programmatic"] == 0
            assert _tile(calls[i + 1][0]) and calls[i + 1][1]["programmatic"] == 1   # the black pass may


# no memory for boundary rows, row sums or partials (mpr_run gave MPR_ERR_OOM): one launch per pass, the energy
# partials of each sweep summed before the next
@pytest.mark.parametrize("shape", [(100, 80), (300, 300), (777, 523), (1400, 1200), (4096, 300)])
@pytest.mark.parametrize("func", [0, 1])
def test_runs_without_memory_for_scratch(driver, shape, func):
    status, calls = driver("scarce", *shape, 5, 30, func)
    assert status == 0
    sums = [i for i, (n, _) in enumerate(calls) if "sweep_sums_kernel" in n]
    passes = [i for i, (n, _) in enumerate(calls) if _tile(n) or "12sweep_kernel" in n]
    assert len(sums) == 30 and all(len([p for p in passes if p < s]) % 2 == 0 for s in sums)
    assert len(passes) + 2 * sum(_resident(n) for n, _ in calls) * 5 == 2 * 35


# a single column of at most 32 half-columns runs in 32-column tiles, which have no half-height form
@pytest.mark.parametrize("shape", [(2, 40), (28, 50000), (64, 64), (64, 20000)])
def test_narrow_grids_run_whole_tiles(driver, shape):
    status, calls = driver("run", *shape, 3, 0, 0)
    assert status == 0 and [a["grid"] for n, a in calls if _tile(n)] == 6 * [-(-shape[1] // 32)]
    _, calls = driver("run", 66, shape[1], 3, 0, 0)
    assert all(a["grid"] > -(-shape[1] // 32) for n, a in calls if _tile(n))   # a 64-column tile has halves


# shapes and the fewest plain and measured sweeps that run resident: a cluster in one column of narrow tiles, a
# grid there, a tall one, others
@pytest.mark.parametrize("shape,plain,measured", [((64, 64), 4, 2), ((3, 3), 4, 2), ((60, 400), 3, 2),
                                                  ((60, 20000), 4, 4), ((12, 100000), 2, 2), ((128, 128), 2, 2),
                                                  ((256, 256), 2, 2), ((777, 523), 2, 2), ((1400, 1200), 2, 2)])
def test_short_runs_take_the_quicker_kernel(driver, shape, plain, measured):
    for n in (1, 2, 3, 4, 5):
        for least, call in ((plain, (n, 0)), (measured, (0, n))):
            status, calls = driver("run", *shape, *call)
            assert status == 0 and any(_resident(name) for name, _ in calls) == (n >= least)
            assert any(_tile(name) for name, _ in calls) == (n < least)


# runs in flight (this one included) up to which a lattice runs resident
@pytest.mark.parametrize("shape,most", [((64, 64), 9), ((200, 150), 9), ((256, 256), 9), ((400, 300), 3),
                                        ((512, 400), 9), ((777, 523), 2), ((1024, 1024), 2), ((1400, 1200), 1),
                                        ((12, 100000), 9)])
def test_handles_that_run_at_once_share_the_device(driver, shape, most):
    for others in range(9):
        status, calls = driver("busy", *shape, others)
        assert status == 0 and any(_resident(n) for n, _ in calls) == (others + 1 <= most)


# half-height tiles shorten the last wave of a pass that has the device to itself
@pytest.mark.parametrize("shape,most", [((777, 523), 8), ((1400, 1200), 2), ((2000, 1500), 1)])
def test_no_half_height_tiles_where_other_runs_fill_the_device(driver, shape, most):
    tiles = -(-((shape[0] + 1) // 2) // 128) * -(-shape[1] // 32)
    for others in range(9):
        _, calls = driver("busy", *shape, others)
        plain = [a["grid"] for n, a in calls if _tile(n)][:10]
        assert len(plain) in (0, 10) and all((g > tiles) == (others + 1 <= most) for g in plain)


# a grid's boundary rows carry tags that no earlier launch has used since the rows were last cleared
@pytest.mark.parametrize("shape", [(300, 300), (777, 523)])
def test_tags_start_again_with_cleared_rows(driver, shape):
    assert driver("tags", *shape)[0] == 0
