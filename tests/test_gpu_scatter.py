"""The epilogue's separate scatter kernel (lanes are walkers) against the oracle, where its group
sizes and their edges fall: whole and ragged groups, and every excitation degree."""
from __future__ import annotations

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


def _case(n_up, n_dn, n_mo, n_walk, seed):
    return synth.make_workload("scatter", seed, n_up, n_dn, n_up + n_dn, (12, 8, 4), (0.05, 500.0), n_mo, 5000, 4, n_walk,
                               n_unique=(300, 280))


# walkers: groups of 32 (FP64: 16), of 16 (8) with a ragged last one, one more than whole groups;
# 17 electrons and 60 MOs fit groups of 16 (pairs) and 16 (FP64); 12 and 34 groups of 32 and 16
@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("n_up,n_dn,n_mo,n_walk", [(5, 4, 30, 4865), (5, 4, 30, 1001), (12, 11, 34, 2449), (17, 16, 60, 1300)])
def test_separate_scatter(n_up, n_dn, n_mo, n_walk, prec):
    wl = _case(n_up, n_dn, n_mo, n_walk, 31 + n_walk)
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    if prec == pkg.PRECISION_MIXED:
        ctx.set_fallback(1e-7)  # below the test tolerance, as the parity tests of this path
    out = ctx.evaluate(torch.from_numpy(wl.R).to("cuda:0"))
    torch.cuda.synchronize()
    idx = np.unique(np.concatenate([np.arange(8), [n_walk // 2, n_walk - 2, n_walk - 1]]))
    rep = compare({k: v.cpu().numpy()[idx] for k, v in out.items()}, oracle.evaluate(wl, R=wl.R[idx]), **TOL[prec])
    assert rep["ok"], rep
