"""The contraction as residue products on the tensor cores (csrc/mdet_modgemm.cu)
against the sparse FP64 sums and against the oracle.

Expansions dense enough take the residue products; set_tuning(spmm_blocks > 0) selects
the sparse sums on the same context. The kernels launched tell the two apart (8 and 6 per
evaluation without the fallback).
"""
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

KEYS = ("log_abs_psi", "sign", "grad", "lap", "e_local", "status")
TOL = {pkg.PRECISION_FP64: dict(tol_psi=1e-10, tol_der=1e-8), pkg.PRECISION_MIXED: dict(tol_psi=1e-9, tol_der=1e-6)}
SPARSE_GRID = 1 << 20


def _eval(ctx, R):
    out = ctx.evaluate(torch.from_numpy(np.ascontiguousarray(R)).to("cuda:0"))
    torch.cuda.synchronize()
    return {k: out[k].cpu().numpy() for k in KEYS}


def _workload(n_up_det, n_dn_det, n_walk, n_det=None, seed=5):
    """5 up / 4 down electrons in 30 MOs with the given numbers of distinct determinants."""
    n_det = n_det or max(4200, max(n_up_det, n_dn_det) * 3)
    n_det = min(n_det, n_up_det * n_dn_det)
    return synth.make_workload("mod", seed, 5, 4, 9, (12, 6, 2), (0.05, 500.0), 30, n_det, 4, n_walk,
                               n_unique=(n_up_det, n_dn_det))


# distinct determinants around the 64-wide K blocks and the 256-row (and 32-row) tiles
SIZES = [(70, 66), (64, 128), (65, 129), (255, 257), (256, 256), (513, 96)]


@pytest.mark.parametrize("prec", [pkg.PRECISION_FP64, pkg.PRECISION_MIXED])
@pytest.mark.parametrize("nu,nd", SIZES)
def test_residue_products_match_oracle_and_sparse_sums(nu, nd, prec):
    wl = _workload(nu, nd, 40)
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    assert ctx.stats()["n_det_up"] == nu and ctx.stats()["n_det_dn"] == nd
    if prec == pkg.PRECISION_MIXED:
        ctx.set_fallback(1e-7)  # below the test tolerance, as the parity tests of this path
    ref = oracle.evaluate(wl)
    got = _eval(ctx, wl.R)
    rep = compare(got, ref, **TOL[prec])
    assert rep["ok"], rep
    ctx.set_fallback(0.0)
    table = _eval(ctx, wl.R)
    assert ctx.last_kernels == 8
    ctx.set_tuning(spmm_blocks=SPARSE_GRID)
    sparse = _eval(ctx, wl.R)
    assert ctx.last_kernels == 6
    # both contractions get the same ratios: they may differ by their own rounding only, 2^-53 per term of
    # the two nested sums, amplified like the CI sum itself, and by the rounding of the logarithm
    tol = (nu + nd) * 2.0 ** -53 * np.maximum(ref["kappa"], 1.0) + 4 * np.spacing(np.abs(ref["log_abs_psi"]))
    assert np.all(np.abs(table["log_abs_psi"] - sparse["log_abs_psi"]) <= tol)
    assert np.array_equal(table["sign"], sparse["sign"]) and np.array_equal(table["status"], sparse["status"])


@pytest.mark.parametrize("n_walk", [1, 31, 255, 257, 513, 1301])
def test_ragged_walkers(n_walk):
    wl = _workload(130, 70, n_walk, seed=6 + n_walk)
    ctx = pkg.Context.from_workload(wl, device=0)
    rep = compare(_eval(ctx, wl.R), oracle.evaluate(wl), **TOL[pkg.PRECISION_FP64])
    assert rep["ok"], rep


@pytest.mark.parametrize("prec", [pkg.PRECISION_FP64, pkg.PRECISION_MIXED])
def test_error_estimates_agree(prec):
    """The magnitude sum feeds the error estimate: as BF16 pairs it is within 2^-15 of the
    sparse kernel's (2^-17 per operand there, 2^-20 here)."""
    wl = _workload(200, 150, 300)
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    ctx.set_fallback(1e9)  # estimates on, nothing flagged
    _eval(ctx, wl.R)
    _, dense = ctx.error_estimates(300)
    ctx.set_tuning(spmm_blocks=SPARSE_GRID)
    _eval(ctx, wl.R)
    _, sparse = ctx.error_estimates(300)
    assert np.all(np.abs(dense - sparse) <= 2.0 ** -15 * sparse)


@pytest.mark.parametrize("prec", [pkg.PRECISION_FP64, pkg.PRECISION_MIXED])
def test_walkers_without_finite_ratios(prec):
    """Coincident electrons make the reference singular and every ratio NaN: the outputs and
    status of such walkers agree with the sparse sums', and their neighbours are untouched."""
    wl = _workload(130, 70, 64)
    R = wl.R.copy()
    R[3, 1] = R[3, 0]    # spin up
    R[40, 7] = R[40, 6]  # spin down
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    ctx.set_fallback(0.0)
    clean = _eval(ctx, wl.R)
    dense = _eval(ctx, R)
    ctx.set_tuning(spmm_blocks=SPARSE_GRID)
    sparse = _eval(ctx, R)
    assert np.array_equal(dense["status"], sparse["status"])
    for k in KEYS[:-1]:
        assert np.array_equal(np.isfinite(dense[k]), np.isfinite(sparse[k])), k
    ok = np.ones(64, bool)
    ok[[3, 40]] = False
    for k in ("log_abs_psi", "sign"):  # each walker's Psi~ is summed in a fixed order
        assert np.array_equal(dense[k][ok], clean[k][ok]), k


def test_dense_rows_take_smaller_moduli():
    """A row with more than 2,048 nonzeros needs moduli below 256 for exact accumulators."""
    wl = synth.make_workload("mod", 11, 5, 4, 9, (12, 6, 2), (0.05, 500.0), 30, 2400 * 40, 4, 6, n_unique=(40, 2400))
    ctx = pkg.Context.from_workload(wl, device=0)
    rep = compare(_eval(ctx, wl.R), oracle.evaluate(wl), **TOL[pkg.PRECISION_FP64])
    assert rep["ok"], rep
    assert ctx.last_kernels == 8 + 8  # the residue products, and the full-LU fallback with its own


@pytest.mark.parametrize("prec", [pkg.PRECISION_FP64, pkg.PRECISION_MIXED])
def test_more_than_eighteen_moduli(prec):
    """Rows of 12,000 nonzeros: residues of a modulus p add up to about 12,000 p / 4 a row, so moduli above about
    106 are excluded, and 124.6 bits take at least 19 (counted with 8 % of margin)."""
    limit, moduli, bits = 1.08 * np.sqrt(8 * 2.0 ** 24 / 12000), [], 0.0
    for p in range(256, 15, -1):
        if p <= limit and bits < 124.6 and all(np.gcd(p, q) == 1 for q in moduli):
            moduli.append(p)
            bits += np.log2(p)
    assert len(moduli) > 18
    wl = synth.make_workload("mod", 12, 5, 4, 9, (12, 6, 2), (0.05, 500.0), 30, 12 * 12000, 4, 7, n_unique=(12, 12000))
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    if prec == pkg.PRECISION_MIXED:
        ctx.set_fallback(1e-7)  # below the test tolerance, as the parity tests of this path
    got = _eval(ctx, wl.R)
    rep = compare(got, oracle.evaluate(wl), **TOL[prec])
    assert rep["ok"], rep
    assert ctx.last_kernels == (8 + 8 if prec == pkg.PRECISION_FP64 else 8 + 14)


@pytest.mark.parametrize("n_walk", [5, 300])
def test_full_lu_contraction(n_walk):
    """Every walker through full LU (a tolerance below any estimate): its contraction as residue
    products, against the oracle and against the sparse sums."""
    wl = _workload(130, 70, n_walk)
    ctx = pkg.Context.from_workload(wl, device=0)
    ctx.set_fallback(1e-30, 512)
    got = _eval(ctx, wl.R)
    assert ctx.last_kernels == 8 + 8 and np.all(got["status"] & pkg.WS_FALLBACK)
    ref = oracle.evaluate(wl)
    rep = compare(got, ref, **TOL[pkg.PRECISION_FP64])
    assert rep["ok"], rep
    ctx.set_tuning(spmm_blocks=SPARSE_GRID)
    sparse = _eval(ctx, wl.R)
    assert ctx.last_kernels == 6 + 5
    tol = 200 * 2.0 ** -53 * np.maximum(ref["kappa"], 1.0) + 4 * np.spacing(np.abs(ref["log_abs_psi"]))
    assert np.all(np.abs(got["log_abs_psi"] - sparse["log_abs_psi"]) <= tol)
    assert np.array_equal(got["sign"], sparse["sign"]) and np.array_equal(got["status"], sparse["status"])


def test_reevaluated_walkers_take_the_sparse_sums():
    """A mixed context re-evaluates its flagged walkers by the FP64 tables and the sparse sums, also where
    the evaluation itself takes the residue products: the kernels launched tell, and the walkers agree with
    an FP64 context on the sparse sums up to the order in which Psi~ is added."""
    wl = _workload(130, 70, 200)
    ctx = pkg.Context.from_workload(wl, device=0, precision=pkg.PRECISION_MIXED)
    ctx.set_escalation(pkg.Context.ESCALATE_ALWAYS)
    ctx.set_fallback(1e9)
    _eval(ctx, wl.R)
    _, est = ctx.error_estimates(200)
    ctx.set_fallback(float(np.median(est[:, 0])), 256)  # half the walkers; the FP64 estimates are 64 times smaller
    got = _eval(ctx, wl.R)
    # 8 of the evaluation; list, gather, two for the orbitals, reference, ratios, sums, epilogue, 5 of full LU, scatter
    assert ctx.last_kernels == 8 + 14
    esc = (got["status"] & pkg.WS_ESCALATED != 0) & (got["status"] & pkg.WS_FALLBACK == 0)
    assert esc.sum() > 50
    f64 = pkg.Context.from_workload(wl, device=0)
    f64.set_fallback(0.0)
    f64.set_tuning(spmm_blocks=SPARSE_GRID, mo_impl=1)
    want = _eval(f64, wl.R)
    tol = 200 * 2.0 ** -53 * np.maximum(oracle.evaluate(wl)["kappa"], 1.0) + 4 * np.spacing(np.abs(want["log_abs_psi"]))
    assert np.all(np.abs(got["log_abs_psi"] - want["log_abs_psi"])[esc] <= tol[esc])
    assert np.array_equal(got["sign"][esc], want["sign"][esc])


@pytest.mark.parametrize("prec", [pkg.PRECISION_FP64, pkg.PRECISION_MIXED])
@pytest.mark.parametrize("n_walk", [513, 700])
def test_blocks_of_walkers(n_walk, prec):
    """The residue products in blocks of 256 walkers (a workspace that holds no more), the last one ragged,
    are those of one block to the bit."""
    wl = _workload(130, 70, n_walk)
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    ctx.set_fallback(0.0)
    whole = _eval(ctx, wl.R)
    assert ctx.last_kernels == 8
    ctx.set_workspace(product_bytes=1)
    got = _eval(ctx, wl.R)
    assert ctx.last_kernels == 8 + 2 * 3
    for k in ("log_abs_psi", "sign"):  # each walker's Psi~ is summed in a fixed order
        assert np.array_equal(got[k], whole[k]), k


@pytest.mark.parametrize("full_lu,prec", [(False, pkg.PRECISION_FP64), (True, pkg.PRECISION_FP64), (False, pkg.PRECISION_MIXED)])
def test_mos_of_very_different_scale(full_lu, prec):
    """Psi does not change when a MO is scaled and the coefficients of the products that occupy it are divided
    by the same power of two: every term of every sum is the same number as before, but rows of C and
    ratios now range over 2^48 (four such MOs per spin), which a fixed-point form relative to the largest would
    cut. Both agree within the rounding of the sums."""
    wl = _workload(130, 70, 60)
    ref = _occupied(wl, int(np.argmax(np.abs(wl.ci_coef))))
    odd = np.array([m % 2 == 1 and m not in ref for m in range(wl.n_mo)])
    power = np.array([12 * sum(odd[m] for m in _occupied(wl, k, True)) for k in range(wl.n_det)])
    scaled = dataclasses.replace(wl, mo_coef=wl.mo_coef * np.where(odd, 2.0 ** 12, 1.0), ci_coef=np.ldexp(wl.ci_coef, -power))
    got = []
    for w in (wl, scaled):
        ctx = pkg.Context.from_workload(w, device=0, precision=prec)
        ctx.set_fallback(1e-30 if full_lu else 0.0)
        got.append(_eval(ctx, wl.R))
    want = oracle.evaluate(wl)
    # as in test_residue_products_match_oracle_and_sparse_sums; pairs carry 2^-47 instead of 2^-53
    u = 2.0 ** -53 if prec == pkg.PRECISION_FP64 else 2.0 ** -47
    tol = 200 * u * np.maximum(want["kappa"], 1.0) + 4 * np.spacing(np.abs(want["log_abs_psi"]))
    assert np.all(np.abs(got[0]["log_abs_psi"] - got[1]["log_abs_psi"]) <= tol)
    assert np.array_equal(got[0]["sign"], got[1]["sign"])


def _occupied(wl, k, twice=False):
    """MOs of the two determinants of product k (twice: one entry per electron)."""
    mos = []
    for words in (wl.det_up[k], wl.det_dn[k]):
        mos += [m for m in range(wl.n_mo) if int(words[m // 64]) >> (m % 64) & 1]
    return mos if twice else set(mos)


def test_the_form_depends_on_the_walkers():
    """1.6 % of 700 x 700 filled: residue products for few walkers, sparse sums for many, with the same results."""
    wl = _workload(700, 700, 64, n_det=8000)
    ctx = pkg.Context.from_workload(wl, device=0)
    ctx.set_fallback(0.0)
    few = _eval(ctx, wl.R)
    assert ctx.last_moduli >= 16
    many = _eval(ctx, np.tile(wl.R, (128, 1, 1)))
    assert ctx.last_moduli == 0
    # as in test_residue_products_match_oracle_and_sparse_sums
    tol = 1400 * 2.0 ** -53 * np.maximum(oracle.evaluate(wl)["kappa"], 1.0) + 4 * np.spacing(np.abs(few["log_abs_psi"]))
    assert np.all(np.abs(few["log_abs_psi"] - many["log_abs_psi"][:64]) <= tol)
    assert np.array_equal(few["sign"], many["sign"][:64]) and np.array_equal(few["status"], many["status"][:64])
    again = _eval(ctx, wl.R)
    assert ctx.last_moduli >= 16 and np.array_equal(again["log_abs_psi"], few["log_abs_psi"])


@pytest.mark.parametrize("n_walk", [1217, 1300, 1303])
def test_wide_rows_of_many_walkers(n_walk):
    """As test_mos_of_very_different_scale, with more walkers than eight an SM, which the reconstruction takes
    four to a block (the last block ragged): every fourth of them, and its neighbours, as in a small batch."""
    wl = _workload(130, 70, 64)
    ref = _occupied(wl, int(np.argmax(np.abs(wl.ci_coef))))
    odd = np.array([m % 2 == 1 and m not in ref for m in range(wl.n_mo)])
    power = np.array([12 * sum(odd[m] for m in _occupied(wl, k, True)) for k in range(wl.n_det)])
    scaled = dataclasses.replace(wl, mo_coef=wl.mo_coef * np.where(odd, 2.0 ** 12, 1.0), ci_coef=np.ldexp(wl.ci_coef, -power))
    ctx = pkg.Context.from_workload(scaled, device=0)
    ctx.set_fallback(0.0)
    few = _eval(ctx, wl.R)
    many = _eval(ctx, np.tile(wl.R, (21, 1, 1))[:n_walk])
    assert ctx.last_moduli >= 16
    want = oracle.evaluate(wl)
    tol = 200 * 2.0 ** -53 * np.maximum(want["kappa"], 1.0) + 4 * np.spacing(np.abs(want["log_abs_psi"]))
    at = np.arange(n_walk) % 64
    assert np.all(np.abs(many["log_abs_psi"] - few["log_abs_psi"][at]) <= tol[at])
    assert np.array_equal(many["sign"], few["sign"][at])
    rep = compare(few, want, **TOL[pkg.PRECISION_FP64])
    assert rep["sign_ok"], rep
