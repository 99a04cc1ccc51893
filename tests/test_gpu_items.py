"""The sparse contraction's work items shrink when there are too few to fill the chip: every item
size from 16 up, with whole and cut segments, against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1510_00730_gb300 as pkg
from paper_1510_00730_gb300 import synth
from tests.parity import compare

pytestmark = pytest.mark.gpu

TOL = {pkg.PRECISION_FP64: dict(tol_psi=1e-10, tol_der=1e-8), pkg.PRECISION_MIXED: dict(tol_psi=1e-9, tol_der=1e-6)}


@pytest.mark.parametrize("prec", [pkg.PRECISION_FP64, pkg.PRECISION_MIXED])
@pytest.mark.parametrize("n_det,n_walk", [(60, 3), (300, 520), (3000, 64), (3000, 3000)])
def test_small_contractions(n_det, n_walk, prec):
    wl = synth.oxygen_like_1k(n_walk=n_walk, seed=77)
    order = np.argsort(-np.abs(wl.ci_coef), kind="stable")
    if n_det > wl.n_det:  # a fuller matrix: rows longer than the smallest items
        wl = synth.make_workload("o", 78, 4, 4, 8, (10, 8, 1), (0.05, 5000.0), 20, n_det, 3, n_walk,
                                 coef_law="lognormal", n_unique=(60, 60))
    else:
        wl = synth.subset_products(wl, np.isin(np.arange(wl.n_det), order[:n_det]))
    idx = np.arange(min(n_walk, 40))
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    if prec == pkg.PRECISION_MIXED:
        ctx.set_fallback(1e-7)  # below the test tolerance, as the parity tests of this path
    out = ctx.evaluate(torch.from_numpy(wl.R).to("cuda:0"))
    torch.cuda.synchronize()
    rep = compare({k: v.cpu().numpy()[idx] for k, v in out.items()}, oracle.evaluate(wl, R=wl.R[idx]), **TOL[prec])
    assert rep["ok"], rep


def _grids(fn, kernel):
    """Blocks of every launch of `kernel` while fn runs, from the profiler's trace."""
    import json
    import tempfile

    from torch.profiler import ProfilerActivity, profile

    with tempfile.NamedTemporaryFile(suffix=".json") as f:
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            fn()
            torch.cuda.synchronize()
        p.export_chrome_trace(f.name)
        events = json.load(open(f.name))["traceEvents"]
    return [e["args"]["grid"][0] for e in events if e.get("cat") == "kernel" and kernel in e["name"]]


def test_explicit_item_size_is_used():
    """Only the default item size is shortened for a small expansion: the launches of the sparse sums shrink as
    the caller's size grows."""
    wl = synth.oxygen_like_1k(n_walk=64, seed=77)
    ctx = pkg.Context.from_workload(wl, device=0)
    ctx.set_fallback(0.0)
    R = torch.from_numpy(wl.R).to("cuda:0")
    if not _grids(lambda: ctx.evaluate(R), "k_") and not _grids(lambda: ctx.evaluate(R), "k_"):
        pytest.skip("no kernel records from the profiler")
    blocks = {}
    for chunk in (512, 64, 256, 8192):
        ctx.set_tuning(spmm_chunk=chunk)
        ctx.evaluate(R)
        blocks[chunk] = _grids(lambda: ctx.evaluate(R), "k_spmm_seg")
    assert all(len(b) == 1 for b in blocks.values()), blocks
    assert blocks[512] > blocks[64] > blocks[256] > blocks[8192], blocks


def test_explicit_electron_block_selects_the_cuda_core_orbitals():
    """In FP64 an electron block other than the default asks for the CUDA-core orbital kernel (one launch; the
    digit products and the dot products of small bases have three and two), and so it does in mixed
    precision for a basis beyond what the digit products always served."""
    for prec, shells, counts in ((pkg.PRECISION_FP64, (12, 6, 2), {6: 2, 4: 1, 8: 1}),
                                 (pkg.PRECISION_FP64, (20, 20, 5), {6: 3, 4: 1, 8: 1}),
                                 (pkg.PRECISION_MIXED, (20, 20, 5), {4: 2, 6: 2, 8: 2}),
                                 (pkg.PRECISION_MIXED, (20, 20, 5, 5), {4: 3, 6: 1, 8: 1})):
        wl = synth.make_workload("ec", 5, 3, 2, 5, shells, (0.05, 500.0), 30, 60, 3, 10, n_unique=(12, 10))
        ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
        if prec == pkg.PRECISION_MIXED:
            ctx.set_fallback(1e-7)  # below the test tolerance, as the parity tests of this path
        ref = oracle.evaluate(wl)
        n = {}
        for ec in counts:
            ctx.set_tuning(mo_ec=ec)
            got = {k: v.cpu().numpy() for k, v in ctx.evaluate(torch.from_numpy(wl.R).to("cuda:0")).items()}
            rep = compare(got, ref, **TOL[prec])
            assert rep["ok"], rep
            n[ec] = ctx.last_kernels
        default = 6 if prec == pkg.PRECISION_FP64 else 4
        assert {ec: n[ec] - n[default] + counts[default] for ec in counts} == counts
