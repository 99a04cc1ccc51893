"""The digit products of the orbitals (csrc/mdet_mo_digits.cu) at the edges of their tiles (16-AO
slices, 32-MO chunks, 16-electron blocks, 128-row tiles), both precisions, against the oracle, and
against the CUDA-core products (mo_impl 1) for positions that are not finite."""
from __future__ import annotations

import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1510_00730_gb300 as pkg
from paper_1510_00730_gb300 import synth
from tests.parity import compare

pytestmark = pytest.mark.gpu

PRECISIONS = [pytest.param(pkg.PRECISION_FP64, id="fp64"), pytest.param(pkg.PRECISION_MIXED, id="mixed")]
TOL = {pkg.PRECISION_FP64: dict(tol_psi=1e-10, tol_der=1e-8), pkg.PRECISION_MIXED: dict(tol_psi=1e-9, tol_der=1e-6)}
KEYS = ("log_abs_psi", "sign", "grad", "lap", "e_local", "status")


def _eval(ctx, R):
    out = ctx.evaluate(torch.from_numpy(np.ascontiguousarray(R)).to("cuda:0"))
    torch.cuda.synchronize()
    return {k: out[k].cpu().numpy() for k in KEYS}


def _workload(shells, n_mo, n_walk, n_up=3, n_dn=2, seed=9):
    return synth.make_workload("orb", seed, n_up, n_dn, n_up + n_dn, shells, (0.05, 500.0), n_mo, 60, 3, n_walk,
                               n_unique=(12, 10))


# (shells per l) -> AOs: 16, 17, 48, 112, 113, 160; MOs around the 16- and 32-wide chunks
CASES = [((7, 3, 0), 10, 1), ((8, 3, 0), 17, 5), ((12, 6, 3), 33, 26), ((12, 10, 5, 4), 96, 3), ((13, 10, 5, 4), 97, 31),
         ((20, 20, 5, 5), 129, 7), ((20, 20, 5, 5), 31, 52)]


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("shells,n_mo,n_walk", CASES)
def test_tile_edges(shells, n_mo, n_walk, prec):
    wl = _workload(shells, n_mo, n_walk)
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    if prec == pkg.PRECISION_MIXED:
        ctx.set_fallback(1e-7)  # below the test tolerance, as the parity tests of this path
    rep = compare(_eval(ctx, wl.R), oracle.evaluate(wl), **TOL[prec])
    assert rep["ok"], rep


@pytest.mark.parametrize("prec", PRECISIONS)
def test_positions_that_are_not_finite(prec):
    """A NaN or infinite coordinate: that walker's outputs are as with the CUDA-core products, and
    the other walkers' log|Psi| (summed in a fixed order) is untouched."""
    wl = _workload((20, 20, 5, 5), 70, 40)
    R = wl.R.copy()
    R[4, 1, 2] = np.nan
    R[21, 3, 0] = np.inf
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    ctx.set_fallback(0.0)
    clean, got = _eval(ctx, wl.R), _eval(ctx, R)
    ctx.set_tuning(mo_impl=1)
    plain = _eval(ctx, R)
    assert np.array_equal(got["status"], plain["status"])
    for k in KEYS[:-1]:
        assert np.array_equal(np.isfinite(got[k]), np.isfinite(plain[k])), k
    ok = np.ones(40, bool)
    ok[[4, 21]] = False
    tol = 22 * 2.0 ** -50 * np.maximum(oracle.evaluate(wl)["kappa"], 1.0)  # the sparse sums' atomics, in any order
    assert np.all(np.abs(got["log_abs_psi"] - clean["log_abs_psi"])[ok] <= (tol + 1e-14)[ok])


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("digit_bytes", [1, 400_000])
@pytest.mark.parametrize("n_mo", [31, 33])
def test_blocks_of_walkers(n_mo, digit_bytes, prec):
    """The orbitals in blocks of walkers (one at a time, and an odd few) with odd numbers of electrons and
    MOs, so that every other block's array starts half a 16-byte store later; 160 AOs, whose FP64 orbitals
    take digits."""
    wl = _workload((20, 20, 5, 5), n_mo, 23)
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    if prec == pkg.PRECISION_MIXED:
        ctx.set_fallback(1e-7)  # as in test_tile_edges
    whole = _eval(ctx, wl.R)
    ctx.set_workspace(digit_bytes=digit_bytes)
    got = _eval(ctx, wl.R)
    rep = compare(got, oracle.evaluate(wl), **TOL[prec])
    assert rep["ok"], rep
    assert np.array_equal(got["status"], whole["status"]) and np.array_equal(got["sign"], whole["sign"])


@pytest.mark.parametrize("prec,shells,n_mo", [(pkg.PRECISION_FP64, (20, 20, 5, 0), 31), (pkg.PRECISION_FP64, (20, 20, 5, 5), 96),
                                              (pkg.PRECISION_MIXED, (20, 20, 5, 5), 31), (pkg.PRECISION_MIXED, (20, 20, 5, 5), 129)])
@pytest.mark.parametrize("some", [False, True])
def test_mos_without_the_dominant_aos(prec, shells, n_mo, some):
    """Electrons near the nucleus, where tight s functions set the largest value of every row, in MOs (all, or
    every other one) that have none of them: the digits, cut relative to that value, would lose most of
    their decimal places. Every orbital is to be as accurate as a dot product over its own terms (mo_impl 1),
    within a rounding per AO, so that the outputs agree within 4 K times the estimated error of one
    rounding per orbital."""
    wl = _workload(shells, n_mo, 40)
    mo = wl.mo_coef.copy()
    assert np.all(wl.shell_l[:shells[0]] == 0) and np.all(wl.shell_nprim == 3)
    mo[np.ix_(np.arange(shells[0]), np.arange(0, n_mo, 2 if some else 1))] = 0.0
    alpha = wl.alpha.copy()
    alpha[:3 * shells[0]] *= 1e6  # s functions of exponents up to 5e8, the others up to 500
    wl = dataclasses.replace(wl, mo_coef=mo, alpha=alpha, R=wl.R * 1e-4)
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    ctx.set_fallback(1e30)  # estimates on, nothing flagged
    got = _eval(ctx, wl.R)
    ctx.set_tuning(mo_impl=1)
    want = _eval(ctx, wl.R)
    _, est = ctx.error_estimates(len(wl.R))
    for k in ("grad", "lap"):
        d = np.abs(got[k] - want[k]).reshape(len(wl.R), -1).max(1)
        scale = np.sqrt((want[k] ** 2).reshape(len(wl.R), -1).mean(1))
        assert np.all(d <= 4 * wl.n_ao * est[:, 0] * scale), (k, (d / scale / est[:, 0]).max())
    assert np.array_equal(got["sign"], want["sign"])
