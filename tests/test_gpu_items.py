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
