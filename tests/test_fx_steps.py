"""The integer steps of the FP64 operator on the host (csrc/fx_steps.h through a small C++ program), against
sums in exact arithmetic, at the largest values their bounds admit."""

import math
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    exe = tmp_path_factory.mktemp("fx") / "fx_steps_check"
    src = os.path.join(ROOT, "tests", "native", "fx_steps_check.cpp")
    inc = os.path.join(ROOT, "paper_1712_00143_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + inc, src, "-o", str(exe)], check=True)

    def run(sites):
        """sites: [(unit exponent, links [hops, 3, 3], vectors [hops, 3])] -> complex [site, 3] (None: range)"""
        text = []
        for kexp, links, psi in sites:
            text.append(f"site {len(links)} {kexp}")
            for w, v in zip(links, psi):
                c = np.concatenate([np.asarray(w).reshape(9), np.asarray(v)])
                text.append(" ".join(f"{float(z.real).hex()} {float(z.imag).hex()}" for z in c))
        out = subprocess.run([str(exe)], input="\n".join(text) + "\n", capture_output=True, text=True, check=True)
        res = []
        for line in out.stdout.splitlines():
            f = [float.fromhex(x) for x in line.split()] if line != "range" else None
            res.append(None if f is None else np.array(f[0::2]) + 1j * np.array(f[1::2]))
        assert len(res) == len(sites)
        return res

    return run


def exact(links, psi):
    out = []
    for i in range(3):
        re = im = Fraction(0)
        for w, v in zip(links, psi):
            for j in range(3):
                a, b = Fraction(w[i][j].real), Fraction(w[i][j].imag)
                c, d = Fraction(v[j].real), Fraction(v[j].imag)
                re += a * c - b * d
                im += a * d + b * c
        out.append(complex(float(re), float(im)))
    return np.array(out)


def check(steps, sites):
    """48 products per sum: FP64 itself rounds to within 96 * 2^-53 = 1.1e-14 of (sum over hops of the row's
    norm) x (largest vector's norm)."""
    for (_, links, psi), got in zip(sites, steps(sites)):
        want = exact(links, psi)
        row = np.sqrt((np.abs(np.asarray(links)) ** 2).sum(-1)).sum(0).max()
        size = row * np.sqrt((np.abs(np.asarray(psi)) ** 2).sum(-1)).max()
        assert got is not None and np.abs(got - want).max() <= 1.1e-14 * size, (got, want)


def test_sums_keep_their_value_when_the_unit_is_raised(steps):
    """Rows of sixteen hops with norms that add up to 8.995 units, entries (1 + i) c and aligned vectors: the
    third running sum passes 2^63 before a larger last neighbour raises the unit."""
    sites = []
    for z in (1e-3, 1e-2):
        c = (8.995 - 2 * z * math.sqrt(6)) / 14 / math.sqrt(6)
        for s in (1, -1, 1j, -1j):
            links = np.full((16, 3, 3), s * (1 + 1j) * c)
            links[0] = links[15] = (1 + 1j) * z
            psi = np.full((16, 3), 3.999 + 3.999j)
            psi[0], psi[15] = 1.99 + 1.99j, 7.99 + 7.99j
            sites.append((0, links, psi))
            sites.append((0, links, psi.conj()))
    check(steps, sites)


def test_random_fields(steps):
    rng = np.random.default_rng(5)
    sites = []
    for n in range(40):
        links = rng.normal(size=(16, 3, 3)) + 1j * rng.normal(size=(16, 3, 3))
        links *= 0.4 / np.abs(links).max() * rng.choice([1.0, 1 / 16], size=(16, 1, 1))
        psi = (rng.normal(size=(16, 3)) + 1j * rng.normal(size=(16, 3))) * 2.0 ** rng.integers(-8, 9, size=(16, 1))
        sites.append((0, links, psi))
    check(steps, sites)


# bits of a component that the high word does not hold: nearly all set
LOW = 1.0 + (2.0**52 - 1) * 2.0**-52


@pytest.mark.parametrize("c", [1 - 2.0**-40, 1 - 2.0**-33, 0.95, 0.5, 0.8838834, 0.7216878, 0.51])
@pytest.mark.parametrize("hops", [1, 2, 3, 16])
def test_rows_of_the_largest_entries(steps, c, hops):
    """(1 + i) c in one or all colours, vectors of large low parts: the sum of an entry's parts and a row's
    cross products at their largest."""
    sites = []
    for colours in (1, 3):
        for s in (1, -1, 1j, -1j):
            for v in (LOW, 1.5 * LOW, 1.0 + 0.5 * LOW, 1.999999):
                w = np.zeros((hops, 3, 3), dtype=complex)
                w[:, :, :colours] = s * (1 + 1j) * c
                for q in (v + 1j * v, v - 1j * v):
                    sites.append((9999, w, np.full((hops, 3), q)))
    check(steps, sites)


def _gaussian(rng, *shape):
    return rng.normal(size=shape) + 1j * rng.normal(size=shape)


def _size(links, psi):
    """Sum over hops of (row norm) x (vector norm), per row: what the rounding of FP64 sums scales with."""
    rows = np.sqrt((np.abs(links) ** 2).sum(-1))
    return (rows * np.sqrt((np.abs(psi) ** 2).sum(-1))[:, None]).sum(0)


@pytest.mark.parametrize("small", [0, -3, -7, -10, -20, -40, -90])
@pytest.mark.parametrize("hop", [0, 5, 15])
def test_a_small_matrix_keeps_its_accuracy(steps, small, hop):
    """A vector seen only through a matrix far smaller than the others: six multiply-adds in FP64 are off by at
    most 6 * 2^-53 of (row norm) x (vector norm)."""
    rng = np.random.default_rng(100 + hop - small)
    sites = []
    for _ in range(40):
        links, psi = _gaussian(rng, 16, 3, 3), np.zeros((16, 3), dtype=complex)
        links[hop] *= 2.0**small
        psi[hop] = _gaussian(rng, 3) * 2.0 ** rng.integers(-3, 4)
        sites.append((9999, links, psi))
    for (_, links, psi), got in zip(sites, steps(sites)):
        assert (np.abs(got - exact(links, psi)) <= 6 * 2.0**-53 * _size(links, psi)).all()


@pytest.mark.parametrize("far", [0, 10, 40, 70, 200, 400])
def test_vectors_behind_zero_matrices_do_not_count(steps, far):
    """Zero Naik links and far larger vectors three sites away."""
    rng = np.random.default_rng(far)
    sites = []
    for _ in range(20):
        links, psi = _gaussian(rng, 16, 3, 3), _gaussian(rng, 16, 3)
        links.reshape(4, 4, 3, 3)[:, 2:] = 0.0
        psi.reshape(4, 4, 3)[:, 2:] *= 2.0**far
        sites.append((9999, links, psi))
    for (_, links, psi), got in zip(sites, steps(sites)):
        assert (np.abs(got - exact(links, psi)) <= 48 * 2.0**-53 * _size(links, psi)).all()


def test_not_finite_vectors_take_the_fp64_loop(steps):
    rng = np.random.default_rng(9)
    for bad in (np.nan, np.inf):
        links, psi = _gaussian(rng, 16, 3, 3), _gaussian(rng, 16, 3)
        links[3] = 0.0
        psi[3, 1] = bad
        assert steps([(9999, links, psi)]) == [None]
    zero = np.zeros((16, 3, 3), dtype=complex)
    got = steps([(9999, zero, _gaussian(rng, 16, 3)), (9999, _gaussian(rng, 16, 3, 3), zero[:, 0])])
    assert all(g is None or (g == 0).all() for g in got)  # ("range" with nothing met: the caller stores zeros)


def _su3(rng, n):
    return np.linalg.qr(_gaussian(rng, n, 3, 3))[0]


@pytest.mark.parametrize("kind", ["field", "equal hops", "point", "one component", "wide", "far large", "scaled"])
def test_errors_are_no_larger_than_those_of_fp64_sums(steps, kind):
    """Root mean square over 300 sites of the error against exact sums, this form's and that of one FP64
    multiply-add after the other; 5 % for the sample (600 numbers or more: 3 % each)."""
    rng = np.random.default_rng(17)
    sites = []
    for _ in range(300):
        links, psi = 0.5 * _su3(rng, 16), _gaussian(rng, 16, 3)
        if kind != "equal hops":
            links.reshape(4, 4, 3, 3)[:, 2:] /= 24
        if kind in ("point", "one component"):
            keep = psi[rng.integers(16)].copy()
            if kind == "one component":
                keep[1:] = 0.0
            psi[:] = 0.0
            psi[rng.integers(16)] = keep
        elif kind == "wide":
            psi *= 10.0 ** rng.uniform(-6, 6, size=(16, 1))
        elif kind == "far large":
            psi.reshape(4, 4, 3)[:, 2:] *= 100
        elif kind == "scaled":
            links *= rng.uniform(0.2, 2, size=(16, 1, 1))
        sites.append((9999, links, psi))
    mine, fp64 = steps(sites), steps([(7777, w, v) for _, w, v in sites])
    total = [0.0, 0.0]
    for (_, links, psi), got in zip(sites, zip(mine, fp64)):
        size = Fraction(float(_size(links, psi).max()))
        for i in range(3):
            re = im = Fraction(0)
            for w, v in zip(links[:, i], psi):
                for j in range(3):
                    a, b, c, d = (Fraction(float(x)) for x in (w[j].real, w[j].imag, v[j].real, v[j].imag))
                    re += a * c - b * d
                    im += a * d + b * c
            for k in range(2):
                total[k] += float((Fraction(float(got[k][i].real)) - re) / size) ** 2
                total[k] += float((Fraction(float(got[k][i].imag)) - im) / size) ** 2
    assert math.sqrt(total[0]) <= 1.05 * math.sqrt(total[1]), math.sqrt(total[0] / total[1])
