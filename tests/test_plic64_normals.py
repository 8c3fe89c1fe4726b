"""The FP64 Mixed-Youngs-Centred direction (csrc/plic64.cuh: sums on integers)
decides as the rule evaluated in double: stencils at and near the rule's ties
(rounding residues beside empty and full cells, stencils with mirror symmetries,
thin structures), values far below and above the fractions of a step, infinities
and not-a-numbers.  The header compiled for the host, against the oracle's MYC.

Tolerance per component: the rule's sums of 18 rounded terms with weights of 64
in all are off by at most 18 * 64 * 2^-53 < 2^-42 of the largest value, three
of them over the largest Youngs component in the quotient, for which 2^-39 of
that ratio stands; the quotients themselves round by less than 1e-14."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle as O

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_07463_gb300", "csrc")
SOURCE = """
#include "plic64.cuh"
extern "C" void direction(const double* st, double* m, int n) {
    for (int i = 0; i < n; ++i) vof::myc_direction64(st + 27 * i, m + 3 * i, 0.0);
}
"""


@pytest.fixture(scope="module")
def direction(tmp_path_factory):
    d = tmp_path_factory.mktemp("plic64")
    (d / "host.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-x", "c++",
                    str(d / "host.cpp"), "-o", str(d / "host.so")], check=True)
    fn = ctypes.CDLL(str(d / "host.so")).direction
    ptr = np.ctypeslib.ndpointer(np.float64, flags="C_CONTIGUOUS")
    fn.argtypes, fn.restype = [ptr, ptr, ctypes.c_int], None

    def run(st):
        m = np.empty((len(st), 3))
        fn(np.ascontiguousarray(st), m, len(st))
        norm = np.abs(m).sum(1, keepdims=True)
        return m / np.where(np.isfinite(norm), norm, 1.0)

    return run


def stencils(kind, n, rng):
    one = rng.random((n, 27))
    pick = lambda v: rng.choice(v, (n, 27))  # noqa: E731
    if kind == "random":
        st = one
    elif kind == "quarters":
        st = pick([0.0, 0.25, 0.5, 1.0])
    elif kind == "residues":  # what a sweep leaves: a few ulps beside empty, full and half cells
        st = pick([0.0, 0.0, 0.0, 1.0, 0.5]) + pick([0.0, 0.0, 0.0, 1e-17, -1e-17, 3e-18, 1e-16])
    elif kind == "mirror":
        s = one.reshape(n, 3, 3, 3)
        st = 0.5 * (s + np.flip(s, 1 + rng.integers(3))) + 0.0
    elif kind == "mirror residues":
        s = one.reshape(n, 3, 3, 3)
        st = (0.5 * (s + np.flip(s, 1 + rng.integers(3)))).reshape(n, 27) + pick([0.0, 1e-17, -1e-17, 1e-16, -1e-16])
    elif kind == "diagonal mirror":  # sums that cancel, in another order of rounding
        s = pick([0.0, 0.25, 0.5, 1.0, 0.3, 0.7]).reshape(n, 3, 3, 3)
        st = 0.5 * (s + s.transpose(0, 2, 1, 3))
    elif kind == "isolated":  # one cell among residues of any size
        st = 10.0 ** rng.uniform(-320, -10, (n, 27)) * pick([0.0, 1.0, -1.0])
        st[np.arange(n), rng.integers(27, size=n)] = rng.random(n)
    elif kind == "decades":
        st = 10.0 ** rng.uniform(-300, 0, (n, 27))
    elif kind == "tiny":
        st = one * 10.0 ** -rng.uniform(20, 130, (n, 1))
    elif kind == "huge":
        st = one * 10.0 ** rng.uniform(0, 150, (n, 27)) * pick([1.0, -1.0])
    elif kind == "empty":
        st = np.zeros((n, 27))
    elif kind == "not finite":
        st = pick([0.0, 0.5, 1.0])
        for _ in range(2):
            st[np.arange(n), rng.integers(27, size=n)] = rng.choice([np.nan, np.inf, -np.inf, 0.5], n)
    st = np.array(st, dtype=np.float64).reshape(n, 27)
    st[:, 13] = 0.5
    return st


@pytest.mark.parametrize("kind", ["random", "quarters", "residues", "mirror", "mirror residues", "diagonal mirror",
                                  "isolated", "decades", "tiny", "huge", "empty", "not finite"])
def test_direction_decides_as_the_rule(direction, kind):
    st = stencils(kind, 4000, np.random.default_rng(len(kind)))
    got = direction(st)
    with np.errstate(all="ignore"):
        want = np.array([O.myc(s) for s in st])
        largest = np.abs(np.delete(st, 13, axis=1)).max(1)
        slope = np.array([np.abs(O.youngs(s)).max() for s in st])
        tol = 1e-14 + 2.0 ** -39 * np.where(slope > 0, largest / slope, 0.0)
    tol = np.where(np.isfinite(tol), np.minimum(tol, 1e-6), 1e-14)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    off = np.nan_to_num(np.abs(got - want)).max(1) > tol
    assert not off.any(), (int(off.sum()), st[off][0].tolist(), got[off][0], want[off][0])
