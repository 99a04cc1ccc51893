"""Performance cases of the wavefunction library: what its users have it do.

A case is one call (or one short sequence of calls) through the package's public
entry points, described by plain values:

* ``evaluate``: ``Context.evaluate``, the unit of every Monte Carlo step: Psi, its
  sign, the drift, the Laplacians and the local energy of a batch of walkers;
* ``host``: the same through ``Context.evaluate_host``, host buffers in and out;
* ``batch``: several expansions of uneven size replayed as one CUDA graph
  (``Batch.launch``);
* ``move``: one learned Metropolis move: limited drift, proposal, evaluation at the
  proposed positions, network there, both proposal densities;
* ``train``: one maximum-likelihood training pass of the proposal network (forward,
  loss, backward), with its gradients read back.

The wavefunctions are the generator's (``synth``): an oxygen-like and a
chlorine-like system, the chlorine-like one cut by coefficient magnitude, and
uneven systems of 8 to 34 electrons. A case fixes the wavefunction; the walkers
come from the seed of ``prepare``.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1510_00730_gb300 as pkg
from paper_1510_00730_gb300 import binding, synth

DEVICE = 0
EVAL_KEYS = ("log_abs_psi", "sign", "grad", "lap", "e_local", "status")
# a drift-diffusion time step near 50 % acceptance on the chlorine-like system
TAU = 3e-5


# ---------------------------------------------------------------------------
# the cases

def listed():
    return [
        # A small molecule's expansion with the 64 walkers of one short run: the smallest call,
        # where launches and latency count.
        dict(name="oxygen_1k_mixed_w64", kind="evaluate", system="oxygen", n_det=1000, walkers=64,
             precision="mixed", wf_seed=151000731),
        # The same expansion in full precision with an odd walker count.
        dict(name="oxygen_1k_fp64_w257", kind="evaluate", system="oxygen", n_det=1000, walkers=257,
             precision="fp64", wf_seed=151000731),
        # The ordinary production size: 10^5 products, 4,096 walkers.
        dict(name="chlorine_100k_mixed_w4096", kind="evaluate", system="chlorine", n_det=100_000, walkers=4096,
             precision="mixed", wf_seed=151000732),
        # The same expansion in full precision with a ragged batch.
        dict(name="chlorine_100k_fp64_w1000", kind="evaluate", system="chlorine", n_det=100_000, walkers=1000,
             precision="fp64", wf_seed=151000732),
        # The large expansion of the benchmark, every walker of its step.
        dict(name="chlorine_750k_mixed_w8192", kind="evaluate", system="chlorine", n_det=750_000, walkers=8192,
             precision="mixed", wf_seed=151000733),
        # The largest call: the same in full precision, at that path's own error target.
        dict(name="chlorine_750k_fp64_w8192", kind="evaluate", system="chlorine", n_det=750_000, walkers=8192,
             precision="fp64", wf_seed=151000733),
        # The large expansion cut to its largest coefficients: as many distinct determinants as
        # before, but a sparse matrix of products between them.
        dict(name="chlorine_cut28k_mixed_w8192", kind="evaluate", system="cut", n_det=28_417, walkers=8192,
             precision="mixed", wf_seed=151000733),
        # Many electrons in a large basis (34 electrons, 141 AOs, 103 MOs), a ragged batch.
        dict(name="uneven_34e_mixed_w2161", kind="evaluate", system="uneven", n_det=15_142, walkers=2161, electrons=34,
             aos=141, precision="mixed", wf_seed=15100073400),
        # A driver on the host: positions from and results to host memory.
        dict(name="host_100k_mixed_w2048", kind="host", system="chlorine", n_det=100_000, walkers=2048,
             precision="mixed", wf_seed=151000732),
        # Several expansions of uneven size in one graph launch.
        dict(name="batch_8_mixed", kind="batch", expansions=8, max_det=100_000, precision="mixed", wf_seed=151000734),
        # One learned move of a chain on the 10^5-product wavefunction.
        dict(name="move_100k_mixed_w8192", kind="move", system="chlorine", n_det=100_000, walkers=8192,
             precision="mixed", wf_seed=151000732),
        # One training pass of the proposal network on a minibatch of observed moves.
        dict(name="train_w8192", kind="train", walkers=8192, electrons=17, hidden=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("evaluate", "host", "batch", "move", "train"), (12, 1, 2, 2, 1))[0]
    precision = rng.choice(("mixed", "mixed", "fp64"))
    wf_seed = rng.randrange(1, 1 << 30)
    if kind == "train":
        return dict(kind=kind, walkers=_log_int(rng, 512, 8192), electrons=rng.randint(8, 34),
                    hidden=rng.choice((64, 128, 256)))
    if kind == "batch":
        return dict(kind=kind, expansions=rng.randint(2, 6), max_det=_log_int(rng, 10_000, 100_000),
                    precision="mixed", wf_seed=wf_seed)
    system = rng.choice(("oxygen", "chlorine", "chlorine", "cut", "uneven")) if kind == "evaluate" else "chlorine"
    case = dict(kind=kind, system=system, walkers=_log_int(rng, 16, 8192), precision=precision, wf_seed=wf_seed)
    if system == "oxygen":
        case["n_det"] = _log_int(rng, 200, 3000)
    elif system == "cut":
        case["n_det"] = _log_int(rng, 1000, 200_000)
    elif system == "uneven":
        case.update(n_det=_log_int(rng, 1000, 50_000), electrons=rng.randint(8, 34), aos=rng.randint(60, 160))
        case["walkers"] = min(case["walkers"], 4096)
    else:
        case["n_det"] = _log_int(rng, 2000, 750_000 if kind == "evaluate" else 200_000)
    return case


# ---------------------------------------------------------------------------
# wavefunctions and walkers

@functools.lru_cache(maxsize=8)
def _wavefunction(system, n_det, wf_seed, electrons=0, aos=0):
    """The expansion of a case, with a single placeholder walker."""
    if system == "oxygen":
        return synth.make_workload("oxygen", wf_seed, 4, 4, 8, (10, 8, 1), (0.05, 5000.0), 20, n_det, 3, 1,
                                   coef_law="lognormal")
    if system == "chlorine":
        return synth.make_workload("chlorine", wf_seed, 9, 8, 17, (12, 10, 8, 2), (0.03, 1.0e5), 80, n_det, 4, 1)
    if system == "cut":
        full = _wavefunction("chlorine", 750_000, wf_seed)
        keep = np.zeros(full.n_det, bool)
        keep[np.argsort(-np.abs(full.ci_coef), kind="stable")[:n_det]] = True
        return synth.subset_products(full, keep)
    rng = np.random.default_rng(wf_seed)
    n_mo = max(int(round(0.73 * aos)), (electrons + 1) // 2 + 4)
    return synth.make_workload("uneven", wf_seed, (electrons + 1) // 2, electrons // 2, electrons,
                               synth._shell_counts(rng, aos), (0.03, 1.0e5), n_mo, n_det, 4, 1)


def _wf_of(case):
    return _wavefunction(case["system"], case["n_det"], case["wf_seed"], case.get("electrons", 0), case.get("aos", 0))


@functools.lru_cache(maxsize=4)
def _batch_wfs(expansions, max_det, wf_seed):
    return tuple(synth.batched_uneven(expansions, seed=wf_seed, n_det_range=(1e3, float(max_det))))


def _walkers(wl, n_walk, seed, salt=0):
    return synth.make_walkers(np.random.default_rng([seed, salt]), n_walk, wl.n_elec)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(torch.device("cuda", DEVICE))


def _context(wl, precision):
    return pkg.Context.from_workload(wl, device=DEVICE,
                                     precision=pkg.PRECISION_MIXED if precision == "mixed" else pkg.PRECISION_FP64)


def _moves(case, seed):
    """Observed moves R0 -> R1 of a chain, for the training pass."""
    rng = np.random.default_rng([seed, 5])
    r0 = synth.make_walkers(rng, case["walkers"], case["electrons"])
    return r0, r0 + 0.2 * rng.standard_normal(r0.shape)


def _network(n_elec, hidden, seed):
    return binding.MLP(DEVICE, n_elec, hidden=hidden, seed=1 + seed % 1000, mu_max=1.0, s0=0.5 * math.log(TAU),
                       s_span=1.0, zero_head=False)


# ---------------------------------------------------------------------------
# the calls

def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        r0, r1 = _moves(case, seed)
        mlp = binding.MLP(DEVICE, case["electrons"], hidden=case["hidden"], seed=1 + seed % 1000, s0=-1.5,
                              zero_head=False)
        out = torch.empty(case["walkers"], 4 * case["electrons"], dtype=torch.float32, device="cuda")
        return dict(kind=kind, mlp=mlp, r0=_dev(r0), r1=_dev(r1), out=out, dout=torch.empty_like(out),
                    loss=torch.zeros(1, dtype=torch.float64, device="cuda"))
    if kind == "batch":
        wls = _batch_wfs(case["expansions"], case["max_det"], case["wf_seed"])
        ctxs = [_context(wl, case["precision"]) for wl in wls]
        Rs = [_dev(_walkers(wl, wl.n_walk, seed, i)) for i, wl in enumerate(wls)]
        return dict(kind=kind, batch=binding.Batch(ctxs, Rs, n_streams=8))
    wl = _wf_of(case)
    R = _walkers(wl, case["walkers"], seed)
    ctx = _context(wl, case["precision"])
    if kind == "host":
        return dict(kind=kind, ctx=ctx, R=R)
    if kind == "evaluate":
        return dict(kind=kind, ctx=ctx, R=_dev(R), out=ctx.alloc_outputs(case["walkers"]))
    # move: the chain's current state at R, and the buffers a chain keeps
    Rd = _dev(R)
    cur = ctx.evaluate(Rd)
    mlp = _network(wl.n_elec, 256, seed)
    st = dict(kind=kind, ctx=ctx, mlp=mlp, R=Rd, cur=cur, out0=mlp.forward(Rd), new=ctx.alloc_outputs(len(R)),
              R_new=torch.empty_like(Rd), fb0=torch.empty_like(Rd), fb1=torch.empty_like(Rd),
              lqf=torch.empty(len(R), dtype=torch.float64, device=Rd.device))
    st.update(lqr=torch.empty_like(st["lqf"]), out1=torch.empty_like(st["out0"]))
    return st


def run(state):
    kind = state["kind"]
    if kind == "evaluate":
        return state["ctx"].evaluate(state["R"], out=state["out"])
    if kind == "host":
        return state["ctx"].evaluate_host(state["R"])
    if kind == "batch":
        return state["batch"].launch()
    if kind == "train":
        mlp = state["mlp"]
        mlp.forward(state["r0"], out=state["out"])
        mlp.nll_grad(state["r0"], state["r1"], state["out"], state["dout"], state["loss"])
        mlp.zero_grad()
        mlp.backward(state["dout"])
        return dict(out=state["out"], loss=state["loss"], grads=mlp.grads())
    ctx, mlp, cur, new = state["ctx"], state["mlp"], state["cur"], state["new"]
    binding.vmc_limit_drift(cur["grad"], TAU, 1.0, state["fb0"])
    mlp.propose(state["R"], state["out0"], 12345, 1, state["R_new"], state["lqf"], drift=state["fb0"])
    ctx.evaluate(state["R_new"], out=new)
    mlp.forward(state["R_new"], out=state["out1"])
    binding.vmc_limit_drift(new["grad"], TAU, 1.0, state["fb1"])
    mlp.reverse(state["R"], state["R_new"], state["out1"], state["lqr"], drift_new=state["fb1"])
    return dict(new, R_new=state["R_new"], out1=state["out1"], log_q_fwd=state["lqf"], log_q_rev=state["lqr"])


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _unique(words):
    """Distinct determinants of one spin: (bit strings [n][n_int], product -> determinant)."""
    return np.unique(words, axis=0, return_inverse=True)


def _eval_work(wl, n_walk):
    N, K, M = wl.n_elec, wl.n_ao, wl.n_mo
    nu, nd = (_unique(w)[0].shape[0] for w in (wl.det_up, wl.det_dn))
    per_walker_io = 8 * (3 * N + 1 + 3 * N + N + 1) + 1 + 4
    shared = 16 * wl.n_det + 8 * K * M + 16 * (nu + nd)
    # per walker: AO -> MO products of the value, gradient and Laplacian; the ratio tables; the two
    # contractions over the products; the small determinants and their cofactors (about 60 each)
    flops = 2 * 5 * N * K * M + 2 * M * (wl.n_up ** 2 + wl.n_dn ** 2) + 4 * wl.n_det + 60 * (nu + nd)
    return dict(bytes=n_walk * per_walker_io + shared, flops=n_walk * flops)


def work(case):
    if case["kind"] == "train":
        W, N, H = case["walkers"], case["electrons"], case["hidden"]
        p = 3 * N * H + H * H + 4 * N * H + 2 * H + 4 * N
        return dict(bytes=W * (2 * 24 * N + 16 * N) + 8 * p, flops=6 * W * (3 * N * H + H * H + 4 * N * H))
    if case["kind"] == "batch":
        parts = [_eval_work(wl, wl.n_walk) for wl in _batch_wfs(case["expansions"], case["max_det"], case["wf_seed"])]
        return dict(bytes=sum(p["bytes"] for p in parts), flops=sum(p["flops"] for p in parts))
    wl = _wf_of(case)
    w = _eval_work(wl, case["walkers"])
    if case["kind"] == "move":
        N = wl.n_elec
        w["bytes"] += case["walkers"] * (3 * 24 * N + 16 * N)
        w["flops"] += 2 * case["walkers"] * (3 * N * 256 + 256 * 256 + 4 * N * 256)
    return w


# ---------------------------------------------------------------------------
# the same quantities in plain 64-bit torch: a full LU of every distinct determinant

def _orbitals(wl, R):
    """MO values, gradients and Laplacians [5][W][N][M] of the positions R [W][N][3]."""
    dev = R.device
    cols, p0 = [], 0
    for s in range(len(wl.shell_l)):
        l, k = int(wl.shell_l[s]), int(wl.shell_nprim[s])
        d = R - _dev(wl.nuc_xyz[wl.shell_center[s]])
        x, y, z = d.unbind(-1)
        r2 = (d * d).sum(-1)
        al = torch.tensor(wl.alpha[p0:p0 + k], dtype=torch.float64, device=dev)
        c = torch.tensor(wl.coef[p0:p0 + k], dtype=torch.float64, device=dev)
        p0 += k
        e = torch.exp(-al * r2[..., None]) * c
        f, f1, f2 = e.sum(-1), -(al * e).sum(-1), (al * al * e).sum(-1)
        for a in range(l, -1, -1):
            for b in range(l - a, -1, -1):
                q = (a, b, l - a - b)
                u = [x ** q[0], y ** q[1], z ** q[2]]
                t = (x, y, z)
                P = u[0] * u[1] * u[2]
                dP, lapP = [], torch.zeros_like(P)
                for i in range(3):
                    o = u[(i + 1) % 3] * u[(i + 2) % 3]
                    dP.append(q[i] * t[i] ** (q[i] - 1) * o if q[i] else torch.zeros_like(P))
                    if q[i] > 1:
                        lapP = lapP + q[i] * (q[i] - 1) * t[i] ** (q[i] - 2) * o
                cols.append(torch.stack([P * f] + [dP[i] * f + 2 * t[i] * P * f1 for i in range(3)] +
                                        [lapP * f + P * ((4 * l + 6) * f1 + 4 * r2 * f2)]))
    X = torch.stack(cols, dim=-1)
    return X @ _dev(wl.mo_coef)


def _exact_eval(wl, R):
    """log|Psi|, grad Psi / Psi, Lap Psi / Psi and the local energy in 64 bits."""
    R = _dev(R)
    dev = R.device
    W, N, M = R.shape[0], wl.n_elec, wl.n_mo
    occ, inv_of = [], []
    for words in (wl.det_up, wl.det_dn):
        u, inv = _unique(words)
        bits = (u[:, :, None] >> np.arange(64, dtype=np.uint64)[None, None, :]) & np.uint64(1)
        bits = bits.reshape(u.shape[0], -1)[:, :M]
        n = int(bits[0].sum())
        occ.append(_dev(np.nonzero(bits)[1].reshape(-1, n)))
        inv_of.append(_dev(np.asarray(inv).ravel().astype(np.int64)))
    C = torch.zeros(len(occ[0]), len(occ[1]), dtype=torch.float64, device=dev)
    C[inv_of[0], inv_of[1]] = _dev(wl.ci_coef)
    res = dict(log_abs_psi=torch.empty(W, dtype=torch.float64, device=dev),
               grad=torch.empty(W, N, 3, dtype=torch.float64, device=dev),
               lap=torch.empty(W, N, dtype=torch.float64, device=dev),
               e_local=torch.empty(W, dtype=torch.float64, device=dev))
    per = sum(o.numel() * o.shape[1] for o in occ) * 8 * 6
    step = max(1, min(W, int(24e9 // per)))
    Z = _dev(wl.Z)
    X = _dev(wl.nuc_xyz)
    for w0 in range(0, W, step):
        r = R[w0:w0 + step]
        B = r.shape[0]
        phi = _orbitals(wl, r)
        D, Sinv, scale = [], [], torch.zeros(B, dtype=torch.float64, device=dev)
        for sp, e0, e1 in ((0, 0, wl.n_up), (1, wl.n_up, N)):
            n = e1 - e0
            S = phi[0][:, e0:e1][:, :, occ[sp]].permute(0, 2, 1, 3).reshape(-1, n, n)
            LU, piv, _ = torch.linalg.lu_factor_ex(S)
            diag = LU.diagonal(dim1=-2, dim2=-1)
            swaps = (piv != torch.arange(1, n + 1, device=dev, dtype=piv.dtype)).sum(-1)
            sgn = torch.where(swaps % 2 == 1, -1.0, 1.0).double() * torch.sign(diag).prod(-1)
            ld = diag.abs().log().sum(-1).reshape(B, -1)
            top = ld.max(1).values
            scale += top
            D.append(sgn.reshape(B, -1) * torch.exp(ld - top[:, None]))
            Sinv.append(torch.linalg.lu_solve(LU, piv, torch.eye(n, dtype=torch.float64, device=dev).expand(S.shape)))
            del S, LU
        wt = [D[1] @ C.T, D[0] @ C]
        psi = (D[0] * wt[0]).sum(1)
        G = torch.empty(B, N, 4, dtype=torch.float64, device=dev)
        for sp, e0, e1 in ((0, 0, wl.n_up), (1, wl.n_up, N)):
            n = e1 - e0
            A = Sinv[sp].reshape(B, -1, n, n) * (D[sp] * wt[sp])[:, :, None, None]
            Q = torch.zeros(B, M, n, dtype=torch.float64, device=dev)
            for a in range(n):
                Q.index_add_(1, occ[sp][:, a], A[:, :, a])
            G[:, e0:e1] = torch.einsum("cwim,wmi->wic", phi[1:, :, e0:e1], Q) / psi[:, None, None]
            del A
        ee = (r[:, :, None] - r[:, None]).norm(dim=-1)
        iu = torch.triu_indices(N, N, 1, device=dev)
        v = (1.0 / ee[:, iu[0], iu[1]]).sum(1)
        v = v - (Z / (r[:, :, None] - X).norm(dim=-1)).sum((1, 2))
        if len(Z) > 1:
            jn = torch.triu_indices(len(Z), len(Z), 1, device=dev)
            v = v + (Z[jn[0]] * Z[jn[1]] / (X[jn[0]] - X[jn[1]]).norm(dim=-1)).sum()
        sl = slice(w0, w0 + B)
        res["log_abs_psi"][sl] = scale + psi.abs().log()
        res["grad"][sl] = G[..., :3]
        res["lap"][sl] = G[..., 3]
        res["e_local"][sl] = -0.5 * G[..., 3].sum(1) + v
    return res


def _lu_cost(wl, n_walk):
    return n_walk * sum(_unique(w)[0].shape[0] * n ** 3 for w, n in ((wl.det_up, wl.n_up), (wl.det_dn, wl.n_dn)))


# LU work (determinants x n^3) that the exact values may take: a few seconds
MAX_LU = 3.2e10


def _exact_outputs(wl, R):
    e = _exact_eval(wl, R)
    return {k: e.get(k) for k in EVAL_KEYS}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        r0, r1 = _moves(case, seed)
        N, H = case["electrons"], case["hidden"]
        mlp = binding.MLP(DEVICE, N, hidden=H, seed=1 + seed % 1000, s0=-1.5, zero_head=False)
        p = _dev(mlp.params().astype(np.float64)).requires_grad_(True)  # the drawn weights, the pass's input
        mlp.close()
        sizes = ((3 * N, H), (H,), (H, H), (H,), (H, 4 * N), (4 * N,))
        W1, b1, W2, b2, W3, b3 = (t.reshape(s) for t, s in zip(p.split([math.prod(s) for s in sizes]), sizes))
        x = _dev(r0).reshape(len(r0), -1) / 2.0
        out = torch.tanh(torch.tanh(x @ W1 + b1) @ W2 + b2) @ W3 + b3
        s = -1.5 + 2.0 * torch.tanh(out[:, 3 * N:])
        mu = torch.exp(s)[:, :, None] * torch.tanh(out[:, :3 * N]).reshape(-1, N, 3)
        d2 = ((_dev(r1) - _dev(r0) - mu) ** 2).sum(-1)
        loss = (0.5 * d2 * torch.exp(-2 * s) + 3 * s).sum(1).mean()
        loss.backward()
        return dict(out=out.detach(), loss=loss.detach().reshape(1), grads=p.grad.cpu().numpy())
    if kind == "batch":
        wls = _batch_wfs(case["expansions"], case["max_det"], case["wf_seed"])
        if sum(_lu_cost(wl, wl.n_walk) for wl in wls) > MAX_LU:
            return None
        return [_exact_outputs(wl, _walkers(wl, wl.n_walk, seed, i)) for i, wl in enumerate(wls)]
    if kind == "move":
        return None  # the proposed positions are the pass's own
    wl = _wf_of(case)
    if _lu_cost(wl, case["walkers"]) > MAX_LU:
        return None
    e = _exact_outputs(wl, _walkers(wl, case["walkers"], seed))
    if kind == "host":
        e = {k: None if v is None else v.cpu().numpy() for k, v in e.items()}
    return e
