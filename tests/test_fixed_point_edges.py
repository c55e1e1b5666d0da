"""The fixed-point header at the edges of its ranges, on the CPU: angles of any value (the kernels convert first
and look at the range later), and the doubled argument of the smallest fields that it serves.
"""
import math
import subprocess

import numpy as np
import pytest

from test_fixed_point import CSRC, HARNESS, LD, TWO_PI_LD, _turn_gap


def _build(path, *flags):
    src, exe = path / "h.cpp", path / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++17", *flags, "-I", CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    return str(exe)


def _run(exe, lines):
    r = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return [ln.split() for ln in r.stdout.strip().split("\n")]


def test_any_angle_is_defined(tmp_path):
    try:
        exe = _build(tmp_path, "-fsanitize=undefined", "-fno-sanitize-recover=all")
    except subprocess.CalledProcessError:
        pytest.skip("this compiler has no sanitizer of undefined behaviour")
    xs = [7.4999999, 7.5, 7.6, 7.9999999, math.nextafter(8.0, 0.0), 8.0, 11.0, 15.999999, 16.0, 1e10, 1e300, 1.7e308, -0.0, -1.0, -7.6, -1e300]
    words = [f"{x.hex()}" for x in xs] + ["inf", "-inf", "nan"]
    assert len(_run(exe, [f"t {w} {q.hex()}" for w in words for q in (0.5, 1.0, 1e-3, 1e-300)])) == 4 * len(words)


def test_doubled_argument_of_small_fields(tmp_path):
    """Fields down to 2^-10, and first guesses as far off as 28 fraction bits of the field allow there: 2^-28 in
    each component (5.4e-6 rad at 2^-10), and 1.5e-6 rad of the FP32 arc tangent."""
    exe = _build(tmp_path)
    rng = np.random.default_rng(9)
    rows = []
    for r in (2.0**-10, 2.0**-9, 0.02, 0.1, 1.0):
        for a in list(rng.uniform(-math.pi, math.pi, 400)) + [0.0, math.pi / 2, -math.pi / 2, math.pi]:
            hx, hy = int(r * math.cos(a) * 2.0**60), int(r * math.sin(a) * 2.0**60)
            eps = rng.choice([-1.0, 1.0, rng.uniform(-1, 1)]) * (math.sqrt(2) * 2.0**-28 / r + 1.5e-6)
            half = math.remainder(2 * (math.atan2(hy, hx) + eps), 2 * math.pi) / 2
            rows.append((hx, hy, round(half / (2 * math.pi) * 2**32), r, eps))
    got = _run(exe, [f"a {hx} {hy} {t0}" for hx, hy, t0, _, _ in rows])
    for (hx, hy, _, r, eps), (t,) in zip(rows, got):
        want = np.arctan2(LD(hy), LD(hx)) / TWO_PI_LD * 2
        # products with 58 bits over |h|, the quotient's 2^-45 of the rest, and the cube that its tangent leaves
        tol = 2.0**-55.5 / r + 2.0**-44 * (abs(eps) + 2.0**-31) + 2 / 3 * (abs(eps) + 2.0**-31) ** 3 + 2.0**-58
        assert _turn_gap(t, want) <= tol, (hx, hy, eps)
