"""The reference kernel against the oracle at the block sizes and electron numbers where it can go
wrong: few walkers (256 threads a block) and many (64)."""
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


# rows in groups of four: 1, whole groups, one more and one less; up to the largest number of
# electrons of a spin (a full warp of columns); unequal spins
@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("n_up,n_dn", [(1, 1), (4, 3), (5, 2), (9, 8), (17, 16), (32, 31)])
def test_reference_block_sizes(n_up, n_dn, prec):
    n_mo = n_up + 8
    wl = synth.make_workload("reference", 77 + n_up, n_up, n_dn, n_up + n_dn, (8, 6, 3), (0.05, 500.0), n_mo, 40, 2, 4,
                             n_unique=(8, 6))
    R = np.tile(wl.R, (300, 1, 1))  # 1200 walkers: above 4 an SM
    ctx = pkg.Context.from_workload(wl, device=0, precision=prec)
    ctx.set_fallback(0.0)  # the table results themselves
    want = oracle.evaluate(wl, R=wl.R)
    few = {k: v.cpu().numpy() for k, v in ctx.evaluate(torch.from_numpy(wl.R).to("cuda:0")).items()}
    many = {k: v.cpu().numpy() for k, v in ctx.evaluate(torch.from_numpy(R).to("cuda:0")).items()}
    for got in (few, {k: v[:4] for k, v in many.items()}, {k: v[-4:] for k, v in many.items()}):
        rep = compare(got, want, **TOL[prec])
        assert rep["ok"], rep
