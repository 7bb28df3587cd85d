"""The separable form of the energy denominators (csrc/sep_factors.h), compiled on the host: every
weight 2 / (E_c - E_v) from the FP32 factors, entry by entry.

Bound: the elimination stops at a relative 2^-26; each factor is rounded to FP32 (2^-24 relative) and
the terms' sizes add up to at most 3 of the weight (checked below), so an entry is off by at most
2^-26 + 3 * 2 * 2^-24 = 3.7e-7 of itself."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BOUND = 2.0 ** -26 + 6.0 * 2.0 ** -24


@pytest.fixture(scope="module")
def factors():
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    out_dir = os.path.join(ROOT, "tests", "_build")
    os.makedirs(out_dir, exist_ok=True)
    so = os.path.join(out_dir, "libsep_check.so")
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1810_07772_gb300", "csrc"), os.path.join(ROOT, "tests", "sep_check.cpp"),
                    "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def call(Ev, Ec, max_terms=64):
        nv, nc = len(Ev), len(Ec)
        E = np.concatenate([Ev, Ec]).astype(np.float64)
        cap = max_terms * (nv + nc + 32)
        tab, scale, ldu = np.zeros(cap, np.float32), np.zeros(max_terms, np.float32), ctypes.c_int()
        T = lib.sep_check(E.ctypes.data_as(ctypes.c_void_p), nv, nc, max_terms, ctypes.byref(ldu),
                          tab.ctypes.data_as(ctypes.c_void_p), scale.ctypes.data_as(ctypes.c_void_p),
                          ctypes.c_long(cap))
        assert T >= 0
        tab = tab[: T * ldu.value].reshape(T, ldu.value).astype(np.float64)
        cpad = (nc + 15) // 16 * 16
        return T, tab[:, :cpad], tab[:, cpad:], scale[:T].astype(np.float64)

    return call


def _energies(kind, nv, nc, rng):
    if kind == "uniform":            # the workloads' energies, in Hartree
        return rng.uniform(-10, 0, nv) / 27.2, rng.uniform(0.5, 20, nc) / 27.2
    if kind == "metal":              # a gap of 1e-4 of the band width
        return -rng.random(nv) ** 3, 1e-4 + rng.random(nc) ** 3
    if kind == "degenerate":         # shells of equal energies
        return np.round(rng.uniform(-4, 0, nv)) / 4 - 0.1, np.round(rng.uniform(0, 8, nc)) / 4 + 0.1
    return np.full(nv, -0.3), np.full(nc, 0.2)   # one denominator


@pytest.mark.parametrize("nv,nc", [(1, 1), (1, 40), (16, 16), (17, 97), (32, 480), (64, 1000)])
@pytest.mark.parametrize("kind", ["uniform", "metal", "degenerate", "one"])
def test_every_weight(factors, kind, nv, nc):
    rng = np.random.default_rng(nv + 7 * nc)
    Ev, Ec = _energies(kind, nv, nc, rng)        # not sorted: the library takes any order
    T, z, u, scale = factors(Ev, Ec)
    assert 1 <= T <= min(nv, nc)
    if kind == "one":
        assert T == 1
    if kind == "uniform":
        assert T <= 13
    assert np.abs(z).max() <= 1 and np.abs(u).max() <= 1
    assert not z[:, nc:].any() and not u[:, nv:].any()          # padding
    w = 2.0 / (Ec[None, :] - Ev[:, None])
    terms = np.einsum("t,tv,tc->tvc", scale, u[:, :nv], z[:, :nc][:, ::-1])   # z runs from the last state down
    assert np.max(np.abs(terms).sum(axis=0) / w) <= 3
    got = terms.sum(axis=0)
    assert np.max(np.abs(got - w) / w) <= BOUND


def test_out_of_terms_or_range(factors):
    rng = np.random.default_rng(5)
    Ev, Ec = _energies("uniform", 32, 480, rng)
    T, *_ = factors(Ev, Ec)
    assert factors(Ev, Ec, max_terms=T)[0] == T
    assert factors(Ev, Ec, max_terms=T - 1)[0] == 0             # the caller takes the pair form
    assert factors(Ev * 1e-40, Ec * 1e-40)[0] == 0              # scales that FP32 cannot carry
