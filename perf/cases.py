"""The work a user has the library do, as cases that can be timed and compared.

Every case goes through the public Python entry points: runs of leapfrog steps
(``Context.step`` and ``Batch.step``), measurements (``Context.energy`` with
``Context.observables``), trial samples (``Context.trial_orbitals``) and the
entry point that allocates nothing (``local_energy_noalloc``).  The sizes are
those of the repository's workloads (8, 50, 120 and 200 orbitals), of its tests
(37 orbitals with 7 + 5 electrons) and of its uneven batches (40 to 120
orbitals); the largest workloads keep their systems and paths and carry fewer
walkers, so that a pass stays below a second.

Systems are synthetic molecules with the distributions of ``afqmc_inputs``,
drawn on the GPU.  A measurement's walkers and paths are made here in plain
torch and loaded into the context, so that their values do not depend on the
library.  A run resumes a checkpoint of the library's own burnt-in initial state,
takes a block of steps and writes the checkpoint that ends it, so that every pass
does the same work (left to run on, a synthetic molecule's signs decay and the
work drifts); the cached form, whose cache a checkpoint does not hold, runs on.
"""

import math

import numpy as np
import torch

from paper_2505_18519_gb300 import afqmc as lib

DEV = "cuda"


def listed():
    return [
        # a small run of the plain method (the size checked against full CI): launches and latency count
        dict(name="small_run", kind="run", N=8, n_up=4, n_dn=4, G=32, K=8, W=64, P=16, steps=10, precision="fp64",
             rcache=False, proposal="prior"),
        # the medium molecule's FP64 run, the library's default options, whole population
        dict(name="medium_run", kind="run", N=50, n_up=10, n_dn=10, G=250, K=50, W=512, P=32, steps=1,
             precision="fp64", rcache=False, proposal="prior"),
        # the same molecule with the half-rotated matrices cached from step to step, half the population
        dict(name="medium_run_cached", kind="run", N=50, n_up=10, n_dn=10, G=250, K=50, W=256, P=32, steps=1,
             precision="fp64", rcache=True, proposal="prior"),
        # measuring a checkpoint of the medium run: energy, overlaps and force bias of every pair
        dict(name="medium_energy", kind="energy", N=50, n_up=10, n_dn=10, G=250, K=50, W=512, P=32,
             precision="fp64"),
        # a small open-shell system with odd sizes and few, odd paths
        dict(name="ragged_energy", kind="energy", N=37, n_up=7, n_dn=5, G=40, K=12, W=24, P=9, precision="fp64"),
        # the FP64 measurement that the mixed path of the large molecule is compared with, on some walkers
        dict(name="large_energy_fp64", kind="energy", N=120, n_up=24, n_dn=24, G=600, K=120, W=8, P=64,
             precision="fp64"),
        # the largest molecule measured on the mixed path (three-part FP16 operands, refinement on)
        dict(name="largest_energy_mixed", kind="energy", N=200, n_up=40, n_dn=40, G=1000, K=200, W=32, P=16,
             precision="fp16x6"),
        # the large molecule's mixed run
        dict(name="large_run_mixed", kind="run", N=120, n_up=24, n_dn=24, G=600, K=120, W=64, P=64, steps=4,
             precision="fp16x6", rcache=False, proposal="prior"),
        # the medium molecule's mixed run with the learned proposal, trained online
        dict(name="medium_run_learned", kind="run", N=50, n_up=10, n_dn=10, G=250, K=50, W=512, P=32, steps=2,
             precision="fp16x3", rcache=False, proposal="mlp"),
        # several molecules of uneven size stepped together by one graph
        dict(name="uneven_batch", kind="batch", sizes="40,75,95,120", W=32, P=16, steps=1, precision="fp16x6"),
        # energies of a batch of pairs for a caller that must not allocate
        dict(name="pairs_noalloc", kind="noalloc", N=50, n_up=10, n_dn=10, G=250, pairs=1024, per_walker=32),
        # trial samples for given hidden variables (building or checking a trial)
        dict(name="trial_samples", kind="trial", N=50, n_up=10, n_dn=10, G=250, K=50, samples=4096,
             precision="fp64"),
    ]


# ------------------------------------------------------------------ work
def _measure_flops(N, nu, nd, G, W, P):
    """Y_g = X_g phi per walker, then per pair the overlap, Phi^T Y_g A^-1 and its traces."""
    s2, s3, nt = nu * nu + nd * nd, nu ** 3 + nd ** 3, nu + nd
    pair = (G + 1) * (4 * N * s2 + 8 * s3) + 8 * G * s2 + 4 * N * s2 + 11 * s3
    return W * P * pair + W * (G + 1) * 4 * N * N * nt


def _step_flops(N, nu, nd, G, K, W, P):
    s2, s3, nt = nu * nu + nd * nd, nu ** 3 + nd ** 3, nu + nd
    pair = 2 * (4 * N * s2 + 3 * s3) + 2 * K * N * N + 12 * 2 * N * N * nu   # two overlaps, S, 12 terms of exp(S) Phi0
    return _measure_flops(N, nu, nd, G, W, P) + W * P * pair + W * (4 * G * N * N + 56 * N * N * nt)


def _system_bytes(N, G, K, nu):
    return 8 * ((1 + G + K) * N * N + N * nu)


def _state_bytes(N, nu, nd, K, W, P):
    return 16 * W * N * (nu + nd) + 8 * W + 8 * W * P * (K + N * nu)


def _batch_systems(case):
    return [dict(kind="run", N=N, n_up=N // 5, n_dn=N // 5, G=5 * N, K=N, W=case["W"], P=case["P"],
                 precision=case["precision"], rcache=False, proposal="prior", steps=case["steps"])
            for N in (int(t) for t in case["sizes"].split(","))]


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        parts = [work(s) for s in _batch_systems(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    N, nu, nd, G = c["N"], c["n_up"], c["n_dn"], c["G"]
    if kind == "run":
        K, W, P = c["K"], c["W"], c["P"]
        return {"bytes": _system_bytes(N, G, K, nu) + 2 * _state_bytes(N, nu, nd, K, W, P) + 32 * c["steps"],
                "flops": c["steps"] * _step_flops(N, nu, nd, G, K, W, P)}
    if kind == "energy":
        K, W, P = c["K"], c["W"], c["P"]
        out = 16 * (W + 2 * W * P + W * G)
        return {"bytes": 8 * (1 + G) * N * N + _state_bytes(N, nu, nd, 0, W, P) + out,
                "flops": _measure_flops(N, nu, nd, G, W, P)}
    if kind == "noalloc":
        W, P = c["pairs"] // c["per_walker"], c["per_walker"]
        out = 16 * c["pairs"] * (2 + G)
        return {"bytes": 8 * (1 + G) * N * N + _state_bytes(N, nu, nd, 0, W, P) + out,
                "flops": _measure_flops(N, nu, nd, G, W, P)}
    n, K = c["samples"], c["K"]
    return {"bytes": 8 * (n * K + K * N * N + N * nu + n * N * nu), "flops": n * (2 * K * N * N + 24 * N * N * nu)}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 13)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _symmetric(g, count, N, diag, off):
    a = torch.triu(_normal(g, count, N, N), 1) * off
    a = a + a.transpose(1, 2)
    a.diagonal(dim1=1, dim2=2).copy_(diag)
    return a


def _system(g, N, nu, G, K):
    """h, L, Phi0, U: random symmetric matrices, the lowest eigenvectors of h; the larger
    systems' off-diagonal entries carry 1/sqrt(N)."""
    s = 1.0 / math.sqrt(N) if N >= 20 else 1.0
    h = _symmetric(g, 1, N, -2.0 * torch.rand(1, N, generator=g, device=DEV, dtype=torch.float64), 0.1 * s)[0]
    L = _symmetric(g, G, N, 0.05 * _normal(g, G, N), 0.05 * s)
    U = _symmetric(g, K, N, 0.1 * _normal(g, K, N), 0.1 * s)
    Phi0 = torch.linalg.eigh(h)[1][:, :nu]
    top = Phi0.gather(0, Phi0.abs().argmax(0, keepdim=True))
    return h.contiguous(), L.contiguous(), (Phi0 * top.sign()).contiguous(), U.contiguous()


def _trial_energy(h, L, Phi0, nd):
    """Energy of the determinant Phi0: the constant that keeps a run's weights of order one."""
    e, v = 0.0, torch.zeros(L.shape[0], device=DEV, dtype=torch.float64)
    for C in (Phi0, Phi0[:, :nd]):
        M = C.T @ L @ C
        e += float((C * (h @ C)).sum() - 0.5 * (M * M).sum())
        v += M.diagonal(dim1=1, dim2=2).sum(1)
    return e + 0.5 * float((v * v).sum())


def _trial(Phi0, U, x):
    """exp(sum_k x_k U_k) Phi0 for the rows of x, in 64 bits."""
    out = []
    for part in x.split(1024):
        S = (part @ U.reshape(U.shape[0], -1)).reshape(-1, *U.shape[1:])
        out.append(torch.linalg.matrix_exp(S) @ Phi0)
    return torch.cat(out)


def _states(g, Phi0, U, nd, W, P):
    """Walkers near trial samples of their own, with complex noise as propagation leaves
    it, and paths whose variables are correlated with their walker's."""
    N, nu = Phi0.shape
    K = U.shape[0]
    xw = _normal(g, W, K)
    x = 0.6 * xw[:, None, :] + 0.8 * _normal(g, W, P, K)
    Phi = _trial(Phi0, U, x.reshape(W * P, K)).reshape(W, P, N, nu)
    base = _trial(Phi0, U, xw)

    def walkers(n):
        noise = 0.2 / math.sqrt(N) * torch.complex(_normal(g, W, N, n), _normal(g, W, N, n))
        A = base[:, :, :n] / base[:, :, :n].norm(dim=1, keepdim=True) + noise
        C = torch.linalg.cholesky(A.mH @ A)
        return torch.linalg.solve_triangular(C, A.mH.contiguous(), upper=False).mH.contiguous()

    up = walkers(nu)
    dn = walkers(nd) if nd else torch.zeros(W, N, 0, device=DEV, dtype=torch.complex128)
    weight = torch.exp(0.3 * _normal(g, W))
    return up, dn, weight, x, Phi


def _config(c, W, P, seed, **more):
    kw = dict(n_burn=10, precision=c["precision"], history_capacity=64)
    kw.update(more)
    tau = 0.01 if c["N"] < 20 else 0.005
    return lib.make_config(c["N"], c["n_up"], c["n_dn"], c["G"], c["K"], W, P, tau, 1000003 * int(seed) + 17, **kw)


def _run_context(c, seed, stream=None, salt=0):
    g = _gen(seed * 31 + salt)
    h, L, Phi0, U = _system(g, c["N"], c["n_up"], c["G"], c["K"])
    cfg = _config(c, c["W"], c["P"], seed * 31 + salt, e_shift=_trial_energy(h, L, Phi0, c["n_dn"]), pop_period=5,
                  rcache=c["rcache"], proposal=c["proposal"], mlp_train=c["proposal"] == "mlp")
    return lib.Context(cfg, h, L, Phi0, U, stream=stream)


def _energy_inputs(c, seed):
    g = _gen(seed)
    system = _system(g, c["N"], c["n_up"], c["G"], c["K"])
    return system, _states(g, system[2], system[3], c["n_dn"], c["W"], c["P"])


def _noalloc_inputs(c, seed):
    g = _gen(seed)
    h, L, Phi0, U = _system(g, c["N"], c["n_up"], c["G"], c["N"])
    W = c["pairs"] // c["per_walker"]
    up, dn, _, _, Phi = _states(g, Phi0, U, c["n_dn"], W, c["per_walker"])
    return h, L, Phi.reshape(c["pairs"], c["N"], c["n_up"]).contiguous(), torch.cat([up, dn], dim=2).contiguous()


def _trial_inputs(c, seed):
    g = _gen(seed)
    system = _system(g, c["N"], c["n_up"], c["G"], c["K"])
    return system, _normal(g, c["samples"], c["K"])


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "run":
        ctx = _run_context(c, seed)
        return dict(kind=kind, steps=c["steps"], ctx=ctx, start=None if c["rcache"] else ctx.save_state())
    if kind == "batch":
        ctxs = [_run_context(s, seed, stream=torch.cuda.Stream(), salt=1 + i)
                for i, s in enumerate(_batch_systems(c))]
        torch.cuda.synchronize()
        return dict(kind=kind, steps=c["steps"], ctxs=ctxs, batch=lib.Batch(ctxs),
                    starts=[ctx.save_state() for ctx in ctxs])
    if kind == "energy":
        (h, L, Phi0, U), (up, dn, weight, x, Phi) = _energy_inputs(c, seed)
        ctx = lib.Context(_config(c, c["W"], c["P"], seed, n_burn=0), h, L, Phi0, U)
        ctx.load_state_arrays(dict(step=0, phi_up=up.cpu().numpy(), phi_dn=dn.cpu().numpy(),
                                   weight=weight.cpu().numpy(), x=x.cpu().numpy(), Phi=Phi.cpu().numpy()))
        return dict(kind=kind, ctx=ctx)
    if kind == "noalloc":
        h, L, Phi, phi = _noalloc_inputs(c, seed)
        n = c["pairs"]
        out = [torch.empty(2 * k, dtype=torch.float64, device=DEV) for k in (n, n, n * c["G"])]
        return dict(kind=kind, dims=(c["N"], c["n_up"], c["n_dn"], c["G"], n, c["per_walker"]),
                    args=(h, L, Phi, torch.view_as_real(phi).contiguous()), out=out)
    (h, L, Phi0, U), x = _trial_inputs(c, seed)
    ctx = lib.Context(_config(c, c["samples"], 1, seed, n_burn=0), h, L, Phi0, U)
    return dict(kind=kind, ctx=ctx, x=x.cpu().numpy())


# ------------------------------------------------------------------ one pass
def _state(ctx, steps):
    out = ctx.state_arrays()
    out["history"] = ctx.history(steps)
    return out


def run(state):
    kind = state["kind"]
    if kind == "run":
        if state["start"] is not None:
            state["ctx"].load_state(state["start"])
        state["ctx"].step(state["steps"])
        return _state(state["ctx"], state["steps"])
    if kind == "batch":
        for ctx, start in zip(state["ctxs"], state["starts"]):
            ctx.load_state(start)
        state["batch"].step(state["steps"])
        state["batch"].sync()
        return [_state(c, state["steps"]) for c in state["ctxs"]]
    if kind == "energy":
        out = state["ctx"].energy(walkers=True)
        out.update(state["ctx"].observables())
        return out
    if kind == "noalloc":
        lib.local_energy_noalloc(*state["dims"], *state["args"], *state["out"])
        return state["out"]
    return state["ctx"].trial_orbitals(state["x"])


# ------------------------------------------------------------------ 64-bit values
def _pair_values(h, L, Phi, phi_up, phi_dn):
    """log-overlap, local energy and force-bias values of every pair, from their
    definition: Theta = phi (Phi^T phi)^-1, M_g = Phi^T X_g Theta, one walker at a time."""
    W, P, N, _ = Phi.shape
    G = L.shape[0]
    X = torch.cat([h[None], L]).reshape((G + 1) * N, N)
    logov = torch.empty(W, P, dtype=torch.complex128, device=DEV)
    e = torch.empty(W, P, dtype=torch.complex128, device=DEV)
    v = torch.empty(W, P, G, dtype=torch.complex128, device=DEV)
    for w in range(W):
        lo, tr, ex = 0.0, 0.0, 0.0
        for phi in (phi_up[w], phi_dn[w]):
            n = phi.shape[1]
            if n == 0:
                continue
            F = Phi[w, :, :, :n].transpose(1, 2).contiguous()                  # P, n, N
            A = (F @ phi.real) + 1j * (F @ phi.imag)
            sign, logabs = torch.linalg.slogdet(A)
            lo = lo + torch.complex(logabs, torch.angle(sign))
            Ainv = torch.linalg.inv(A)
            Y = torch.stack([X @ phi.real, X @ phi.imag]).reshape(2, G + 1, N, n)
            Y = Y.permute(2, 0, 1, 3).reshape(N, -1)                           # N, (re/im, g, b)
            for p in range(0, P, 16):
                Z = (F[p:p + 16].reshape(-1, N) @ Y).reshape(-1, n, 2, G + 1, n)
                Z = torch.complex(Z[:, :, 0], Z[:, :, 1]).permute(0, 2, 1, 3)  # pairs, g, a, b
                M = Z @ Ainv[p:p + 16, None]
                t = M.diagonal(dim1=2, dim2=3).sum(2)
                x = (M * M.transpose(2, 3)).sum((2, 3))
                if p == 0:
                    ts, xs = [], []
                ts.append(t)
                xs.append(x)
            tr, ex = tr + torch.cat(ts), ex + torch.cat(xs)
        logov[w] = lo
        v[w] = tr[:, 1:]
        e[w] = tr[:, 0] + 0.5 * (v[w] * v[w] - ex[:, 1:]).sum(1)
    return logov, e, v


def _numpy(t):
    return t.cpu().numpy()


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "trial":
        (_, _, Phi0, U), x = _trial_inputs(c, seed)
        return _numpy(_trial(Phi0, U, x))
    if kind == "noalloc":
        h, L, Phi, phi = _noalloc_inputs(c, seed)
        W, P = c["pairs"] // c["per_walker"], c["per_walker"]
        nu = c["n_up"]
        vals = _pair_values(h, L, Phi.reshape(W, P, c["N"], nu), phi[:, :, :nu], phi[:, :, nu:])
        return [torch.view_as_real(t.contiguous()).reshape(-1) for t in vals]
    if kind == "energy":
        (h, L, _, _), (up, dn, weight, _, Phi) = _energy_inputs(c, seed)
        logov, e, v = _pair_values(h, L, Phi, up, dn)
        S = torch.exp(1j * logov.imag)                      # path signs
        sumS = S.sum(1)
        ew = (S * e).sum(1) / sumS
        fb = (S[:, :, None] * v).sum(1) / sumS[:, None]
        sw = float(weight.sum())
        return dict(e_mix=float((weight * ew.real).sum()) / sw, sum_w=sw,
                    mean_sign=float((weight * sumS.abs()).sum()) / (c["P"] * sw), e_walker=_numpy(ew),
                    logov=_numpy(logov), e_local=_numpy(e), force_bias=_numpy(fb))
    return None                                              # a run's random moves have no plain counterpart


# ------------------------------------------------------------------ more cases of the same ranges
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "energy", "energy", "noalloc", "trial", "batch"])
    if kind == "batch":
        sizes = sorted(rng.sample(range(30, 106, 5), rng.randint(2, 4)))
        return dict(kind=kind, sizes=",".join(map(str, sizes)), W=rng.randint(5, 24), P=rng.randint(3, 16),
                    steps=rng.randint(1, 2), precision=rng.choice(["fp16x6", "fp16x3"]))
    precision = "fp64" if kind == "noalloc" else rng.choice(["fp64", "fp64", "fp64", "fp16x6", "fp16x3"])
    N = _log_int(rng, 8, 200)
    n_up = max(1, min(40, int(N * rng.uniform(0.12, 0.4))))
    n_dn = n_up if rng.random() < 0.5 else rng.randint(0, n_up)
    G = max(4, int(N * rng.uniform(2.0, 6.0)))
    K = max(2, int(N * rng.uniform(0.5, 1.2)))
    if kind == "noalloc":
        per_walker = _log_int(rng, 1, 48)
        fit = min(2048, (28 << 20) // (16 * N * (n_up + n_dn) + 32))
        cost = _measure_flops(N, n_up, n_dn, G, 1, per_walker) / per_walker
        W = max(1, min(fit, int(1e11 / cost), _log_int(rng, 32, 2048)) // per_walker)
        return dict(kind=kind, N=N, n_up=n_up, n_dn=n_dn, G=G, pairs=W * per_walker, per_walker=per_walker)
    if kind == "trial":
        n = _log_int(rng, 64, 4096)
        n = max(16, min(n, int(4e10 / (2 * K * N * N + 40 * N * N * n_up))))
        return dict(kind=kind, N=N, n_up=n_up, n_dn=n_dn, G=G, K=K, samples=n, precision=precision)
    P = _log_int(rng, 1, 64)
    cap = 2e11 if precision == "fp64" else 1.5e12
    W = max(2, min(_log_int(rng, 4, 512), int(cap / _step_flops(N, n_up, n_dn, G, K, 1, P)), 12000 // P))
    c = dict(kind=kind, N=N, n_up=n_up, n_dn=n_dn, G=G, K=K, W=W, P=P, precision=precision)
    if kind == "run":
        c.update(steps=1, rcache=False, proposal=rng.choice(["prior", "prior", "pcn", "rw"]))
        # few electrons in a large basis fit the cached form
        if precision == "fp64" and N * n_up <= 500 and rng.random() < 0.3:
            c["rcache"] = True
    return c
