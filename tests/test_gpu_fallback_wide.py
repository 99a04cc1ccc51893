"""The full-LU fallback at the electron numbers where its kernels change (matrix in registers up to 8 a
spin, in shared memory up to 11, four lanes to a determinant from 12): sizes around the groups of four
rows and columns, unequal spins, determinant counts that leave a ragged last group."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_1510_00730_gb300 as pkg
from paper_1510_00730_gb300 import synth
from tests.parity import compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [pytest.param(pkg.PRECISION_FP64, id="fp64"), pytest.param(pkg.PRECISION_MIXED, id="mixed")])
@pytest.mark.parametrize("n_up,n_dn", [(2, 2), (3, 2), (4, 4), (5, 4), (7, 6), (8, 8), (9, 8), (10, 10), (11, 11), (12, 9), (13, 12), (15, 14), (16, 16), (17, 1), (17, 16)])
def test_every_walker_by_full_lu(n_up, n_dn, prec):
    wl = synth.make_workload("wide", 5 + n_up, n_up, n_dn, n_up + n_dn, (9, 6, 2), (0.05, 500.0), n_up + 6, 90, 4, 7,
                             n_unique=(13, 10))
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    if prec == pkg.PRECISION_MIXED:
        ctx.set_escalation(pkg.Context.ESCALATE_ALWAYS)
    ctx.set_fallback(1e-30, max_walkers=32)
    got = {k: v.cpu().numpy() for k, v in ctx.evaluate(torch.from_numpy(wl.R).to("cuda:0")).items()}
    assert np.all(got["status"] & pkg.WS_FALLBACK)
    rep = compare(got, oracle.evaluate(wl), tol_psi=1e-10, tol_der=1e-8)
    assert rep["ok"], rep
