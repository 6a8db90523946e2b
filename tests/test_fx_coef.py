"""The fixed-point pair kernel's coefficients, evaluated on the host over pair
types of all kinds: every contribution that the rule takes in fixed point stays
in the accumulators' range and within a count of the exact force (and 2^-46 of
its magnitude).  No GPU: the number formats of the kernel are plain C++.
"""
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2508_13523_gb300", "csrc")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("fx") / "fx_coef_check")
    subprocess.check_call(["g++", "-O2", "-std=gnu++17", "-I", CSRC, "-x", "c++",
                           os.path.join(HERE, "fx_coef_check.cpp"), "-o", exe])

    def run(rows):
        """rows of (eps, sigma, rc, rcmax, lmax, qq, rc_coul, samples[, dense]): an
        array of (bad, in fixed point, in range, worst / bound, smallest r in fixed point)."""
        text = "\n".join(" ".join(repr(float(v)) for v in r[:7]) + f" {r[7]} {r[8] if len(r) > 8 else 0}"
                         for r in rows)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return np.array([[float(v) for v in line.split()] for line in out.splitlines()])

    return run


def test_stiff_pairs_with_short_cutoffs(check):
    """Forces beyond the accumulators' range at every separation in fixed point's
    reach, cutoffs at and below a power of two: the FP64 path takes them all."""
    rows = [(3850.0, 2.0 ** (-1 / 6), 1.0, 1.0, 20.0, 0.0, 0.0, 2000),
            (2183.0, 1.0, 1.0, 1.0, 20.0, 0.0, 0.0, 2000),
            (1e5, 0.95, 1.0, 1.0, 20.0, 0.0, 0.0, 2000),
            (4e4, 1.99, 2.0, 2.0, 20.0, 0.0, 0.0, 2000)]
    r = check(rows)
    assert (r[:, 0] == 0).all(), r


@pytest.mark.parametrize("coul", [False, True])
def test_sweep_of_pair_types(check, coul):
    rng = np.random.RandomState(11 + coul)
    rows = []
    for _ in range(400):
        rc = 2.0 ** rng.uniform(-3, 4)
        if rng.rand() < 0.3:
            rc = 2.0 ** rng.randint(-2, 4) * (1.0 if rng.rand() < 0.5 else 1.0 - 2.0 ** -rng.randint(3, 50))
        sigma = rc / 10 ** rng.uniform(-0.05, 1.1)
        eps = 10 ** rng.uniform(-6, 6) * sigma
        rcmax = rc * (1.0 if rng.rand() < 0.6 else rng.uniform(1.0, 6.0))
        lmax = max(4.0, 2.0 * rcmax) * rng.uniform(1.2, 40.0)
        qq, rcc = 0.0, 0.0
        if coul:
            qq = 10 ** rng.uniform(-4, 4) * rng.choice([-1, 1]) * sigma * sigma
            rcc = rcmax * rng.uniform(0.3, 1.0)
        rows.append((eps, sigma, rc, rcmax, lmax, qq, rcc, 300, rng.choice([0, 0, 0, 1, 3, 6])))
    r = check(rows)
    bad = np.nonzero(r[:, 0])[0]
    assert len(bad) == 0, [(rows[k], r[k]) for k in bad[:3]]
    assert (r[:, 1] > 0).mean() > 0.3  # the sweep does reach the fixed-point path


def test_lj_units_in_fixed_point(check):
    """eps = sigma = 1: fixed point down to where the force reaches 256."""
    r = check([(1.0, 1.0, 2.5, 2.5, 168.0, 0.0, 0.0, 20000)])
    assert r[0, 0] == 0 and 0.8637 < r[0, 4] < 0.866
    assert abs(r[0, 1] / r[0, 2] - (2.5 - 0.865) / 2.0) < 0.01  # r uniform in 0.5 .. 2.5


@pytest.mark.parametrize("dense", [1, 2, 3, 6])
def test_dense_lists_keep_their_pairs_in_fixed_point(check, dense):
    """Atoms that may have 2^(11 + dense) partners: contributions have to be smaller
    by 2^dense, and only the pairs whose force is not leave fixed point."""
    r = check([(1.0, 1.0, 4.2, 4.2, 60.0, 0.0, 0.0, 20000, dense)])
    f = lambda r: 24.0 * (2.0 * r ** -13 - r ** -7)
    lo, hi = 0.8, 1.12  # (the samples start at 0.2 rc = 0.84)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (lo, mid) if f(mid) < 2.0 ** (8 - dense) else (mid, hi)
    assert r[0, 0] == 0 and hi - 1e-3 < r[0, 4] < hi + 0.005
