"""The workloads that the speed of this library is judged by.

Each case is one call, or one short chain of calls, that a program makes with
the library's public entry points, at the sizes of the repository's own
workloads, serving mix and tests:

  grad    ln psi of a batch and its gradient in the parameters (autograd)
  sweep   Metropolis sweeps of a set of chains (sampling)
  expect  local energies, their statistics and the force (expect_and_grad)
  qgt     (S + eps I) v with the QGT on the fly
  jac     the stored centred Jacobian and (S + eps I) v with it
  solve   the SR system of given samples, direct solvers
  step    one whole VMC + SR step
  symm    one whole step of the symmetric RBM
  tdvp    one whole time step of the complex RBM
  crbm    ln psi, local energies and log-derivatives of the complex RBM
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2112_10526_gb300 import autograd, inputs, nk


def listed():
    return [
        # The smallest call of a gradient-based program: a few hundred samples
        # of the 16-site Ising chain, forward and backward, default precision.
        dict(name="grad_chain16_f64", op="grad", model="tfim_chain", L=16, alpha=1, B=256, precision="f64", sigma=0.1),
        # Sampling of the 10 x 10 Heisenberg lattice (1024 chains, exchange
        # moves, 16 discarded sweeps and 8 samples a chain).
        dict(name="sweep_heis10_mixed", op="sweep", model="heis_square", L=10, alpha=2, rule="exchange", C=1024,
             n_discard=16, n_samples=8, precision="mixed", sigma=0.05),
        # Energy and force of the 20 x 20 Ising lattice, one sample a chain.
        dict(name="expect_tfim20_mixed", op="expect", model="tfim_square", L=20, alpha=4, Ns=16384, precision="mixed",
             sigma=0.01),
        # Energy and force of the 10 x 10 J1-J2 lattice in full precision.
        dict(name="expect_j1j2_10_f64", op="expect", model="j1j2_square", L=10, alpha=2, Ns=1024, precision="f64",
             sigma=0.05),
        # The product that conjugate gradients repeat on the 24 x 24 lattice:
        # the largest of the configurations, 2.66 M parameters.
        dict(name="qgt_heis24_mixed", op="qgt", model="heis_square", L=24, alpha=8, Ns=65536, precision="mixed",
             sigma=0.01),
        # The same product in full precision (the binding's default), on the
        # 12 x 12 lattice of the serving mix.
        dict(name="qgt_heis12_f64", op="qgt", model="heis_square", L=12, alpha=2, Ns=4096, precision="f64", sigma=0.02),
        # The stored-Jacobian QGT at the ragged sizes of the tests.
        dict(name="jac_ragged_f64", op="jac", model="tfim_chain", L=37, M=45, Ns=1025, precision="f64", sigma=0.1),
        # The direct SR solve of the 10 x 10 Heisenberg workload: Np = 20300
        # parameters through the 8192 x 8192 sample-space matrix.
        dict(name="solve_heis10_mixed", op="solve", model="heis_square", L=10, alpha=2, Ns=8192,
             solver="cholesky_samplespace", precision="mixed", sigma=0.05),
        # The quick-start run: a whole step on the 16-site Ising chain, dense
        # Cholesky, default precision.
        dict(name="step_chain16_f64", op="step", model="tfim_chain", L=16, alpha=1, rule="local", C=16, n_discard=16,
             n_samples=64, solver="cholesky", precision="f64", sigma=0.01),
        # A whole step of the symmetric RBM on the 10 x 10 lattice (4 features
        # over the 100 translations).
        dict(name="symm_heis10_mixed", op="symm", model="heis_square", L=10, alpha=4, rule="exchange", C=1024,
             n_discard=16, n_samples=8, precision="mixed", sigma=0.01),
        # The quench of the 20-site Ising chain: one real-time Heun step.
        dict(name="tdvp_chain20", op="tdvp", model="tfim_chain", L=20, alpha=1, rule="local", C=1024, n_discard=16,
             n_samples=4, integrator="heun", real_time=True, solver="svd", sigma=0.05),
        # The headline: a whole step on the 24 x 24 Heisenberg lattice with
        # conjugate gradients.
        dict(name="step_heis24_mixed", op="step", model="heis_square", L=24, alpha=8, rule="exchange", C=8192,
             n_discard=16, n_samples=8, solver="cg", precision="mixed", sigma=0.01),
    ]


# ------------------------------------------------------------------ sizes ---

def _sites(case):
    return case["L"] ** 2 if "square" in case["model"] else case["L"]


def _hidden(case):
    return case["M"] if "M" in case else case["alpha"] * _sites(case)


def _ham(case):
    return getattr(inputs, case["model"])(case["L"])


def _sz0(case):
    return "tfim" not in case["model"]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _lattice(rng, nmax, square_only=False):
    """A lattice of at most nmax sites: a chain, or a square lattice with even
    side (S_z = 0 and the two sublattices need it)."""
    model = rng.choice(["tfim_square", "heis_square", "j1j2_square"] if square_only else
                       ["tfim_chain", "heis_chain", "tfim_square", "heis_square", "j1j2_square"])
    if "square" in model:
        L = _log_int(rng, 4, int(math.isqrt(nmax)))
    else:
        L = _log_int(rng, 8, nmax)
    if "tfim" not in model:
        L += L % 2
        while (L * L if "square" in model else L) > nmax:
            L -= 2
    return dict(model=model, L=L)


def _limit(rng, n, cost, most):
    """n, made smaller until n * cost stays below most."""
    top = max(16, int(most / max(cost, 1.0)))
    return n if n <= top else _log_int(rng, max(16, top // 8), top)


def draw(rng):
    """One more case of the same ranges: lattices of 8 to 576 sites, 1 to 8
    hidden units a site (odd widths among them), 16 to 65536 samples, both
    precisions, every rule and solver."""
    op = rng.choice(["grad", "sweep", "expect", "qgt", "jac", "solve", "step", "symm", "tdvp", "crbm"])
    precision = rng.choice(["f64", "mixed"])
    slow = 40.0 if precision == "f64" else 1.0  # FP64 runs at about this fraction of the mixed rate
    sigma = rng.choice([0.01, 0.02, 0.05])
    if op in ("grad", "expect", "qgt"):
        case = dict(op=op, **_lattice(rng, 576), precision=precision, sigma=sigma)
        N = _sites(case)
        M = _log_int(rng, N, 8 * N)
        per = 4.0 * N * M * (N if op == "expect" else 1)
        n = _limit(rng, _log_int(rng, 16, 65536), per * slow, 4e12)
        case.update(M=M, **({"B": n} if op == "grad" else {"Ns": n}))
        return case
    if op == "sweep":
        case = dict(op=op, **_lattice(rng, 576), precision=precision, sigma=sigma)
        N = _sites(case)
        M = _log_int(rng, N, 8 * N)
        nd, ns = rng.randint(0, 16), rng.randint(1, 16)
        C = _limit(rng, _log_int(rng, 16, 16384), 2.0 * N * M * (nd + ns) * slow, 1e12)
        rule = rng.choice(["exchange", "hamiltonian"]) if _sz0(case) else "local"
        case.update(M=M, rule=rule, C=C, n_discard=nd, n_samples=ns)
        return case
    if op == "jac":
        case = dict(op=op, **_lattice(rng, 144), precision=precision, sigma=sigma)
        N = _sites(case)
        M = _log_int(rng, N, 4 * N)
        case.update(M=M, Ns=_limit(rng, _log_int(rng, 16, 8192), float(N * M), 4e8))
        return case
    if op == "solve":
        case = dict(op=op, **_lattice(rng, 144), precision=precision, sigma=rng.choice([0.02, 0.05]))
        N = _sites(case)
        M = _log_int(rng, N, 4 * N)
        Np = N + M + N * M
        Ns = _log_int(rng, 64, 8192 if precision == "mixed" else 3000)
        solver = "cholesky" if Np <= (4096 if precision == "mixed" else 2048) else "cholesky_samplespace"
        case.update(M=M, Ns=Ns, solver=solver)
        return case
    if op == "step":
        case = dict(op=op, **_lattice(rng, 256), precision=precision, sigma=sigma)
        N = _sites(case)
        alpha = rng.choice([1, 2, 4])
        M = alpha * N
        Np = N + M + N * M
        nd, ns = rng.randint(0, 16), rng.randint(1, 16)
        C = _limit(rng, _log_int(rng, 16, 1024), 2.0 * N * M * (nd + ns) * slow, 2e11)
        if Np <= 1600:
            solver = "cholesky"
        elif precision == "mixed" and C * ns > 4096:
            solver = "cg"
        else:
            solver = "cholesky_samplespace"
            while C * ns > 4096:
                C //= 2
        rule = rng.choice(["exchange", "hamiltonian"]) if _sz0(case) else "local"
        case.update(M=M, rule=rule, C=C, n_discard=nd, n_samples=ns, solver=solver)
        return case
    if op == "symm":
        case = dict(op=op, **_lattice(rng, 100, square_only=True), precision=precision, sigma=sigma)
        N = _sites(case)
        alpha = rng.randint(1, 4)
        nd, ns = rng.randint(0, 16), rng.randint(1, 8)
        C = _limit(rng, _log_int(rng, 64, 1024), 2.0 * alpha * N ** 3 * (nd + ns) * slow, 4e11)
        case.update(alpha=alpha, rule="exchange" if _sz0(case) else "local", C=C, n_discard=nd, n_samples=ns)
        return case
    if op == "tdvp":
        model = rng.choice(["tfim_chain", "heis_chain"])
        L = rng.randint(10, 20)
        L += L % 2 if model == "heis_chain" else 0
        return dict(op=op, model=model, L=L, alpha=1, rule="exchange" if model == "heis_chain" else "local",
                    C=_log_int(rng, 256, 1024), n_discard=rng.randint(0, 16), n_samples=rng.randint(2, 4),
                    integrator=rng.choice(["euler", "heun"]), real_time=rng.random() < 0.5,
                    solver="svd" if model == "tfim_chain" and rng.random() < 0.5 else "cholesky", sigma=0.05)
    case = dict(op="crbm", **_lattice(rng, 64), sigma=0.05)
    N = _sites(case)
    case.update(M=_log_int(rng, N, 2 * N), Ns=_log_int(rng, 16, 4096))
    return case


# ----------------------------------------------------------------- inputs ---

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _configs(case, n, g):
    """n random configurations: i.i.d. spins, or S_z = 0."""
    N = _sites(case)
    u = torch.rand((n, N), generator=g, device="cuda")
    if _sz0(case):
        u = u.argsort(1).argsort(1) + 0.5 - N / 2
    else:
        u -= 0.5
    return torch.where(u > 0, 1, -1).to(torch.int8)


def prepare(case, seed):
    g = _gen(seed)
    N, ham = _sites(case), _ham(case)
    M = _hidden(case)
    op = case["op"]
    st = SimpleNamespace(case=case, N=N, M=M, ctx=nk.Ctx(), seed=int(seed) % (1 << 40))
    st.edges = torch.from_numpy(ham["edges"]).cuda()
    st.ham = nk.make_ham(ham["kind"], ham["J"], ham["h"], ham["marshall"], st.edges, ham.get("J2", 0.0),
                         ham.get("n_edges2", 0))

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)

    Np = N + M + N * M
    if op == "symm":
        st.perms = torch.from_numpy(inputs.translations_square(case["L"]).astype(np.int32)).cuda()
        st.params = case["sigma"] * normal(1 + case["alpha"] * (1 + N))
    elif op in ("tdvp", "crbm"):
        st.params = case["sigma"] * torch.complex(normal(Np), normal(Np))
    else:
        st.params = case["sigma"] * normal(Np)
    if op in ("sweep", "step", "symm", "tdvp"):
        st.chains = _configs(case, case["C"], g)
    else:
        st.s = _configs(case, case["B"] if op == "grad" else case["Ns"], g)
    if op == "grad":
        st.g = normal(case["B"])
    if op in ("qgt", "jac"):
        st.v = normal(Np)
    if op == "solve":
        # a force: the covariance of the log-derivatives with random local
        # energies
        _a, b, W = _parts(st.params, N, M)
        sd = st.s.double()
        e = normal(case["Ns"])
        st.F = _jtg(torch.tanh(b + sd @ W.T), sd, 2.0 * (e - e.mean()) / case["Ns"])
    return st


# ------------------------------------------------------------------- runs ---

def _empty(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, device="cuda")


def run(st):
    return globals()["_run_" + st.case["op"]](st, st.case, st.N, st.M)


def _run_grad(st, c, N, M):
    p = st.params.detach().requires_grad_(True)
    lp = autograd.logpsi(p, st.s, N, M, st.ctx, c["precision"])
    (grad,) = torch.autograd.grad(lp, p, st.g)
    return {"logpsi": lp.detach(), "grad": grad}


def _run_sweep(st, c, N, M):
    s = st.chains.clone()
    samples = _empty(c["C"], c["n_samples"], N, dtype=torch.int8)
    lp = _empty(c["C"], c["n_samples"])
    acc = torch.zeros(c["C"], dtype=torch.int64, device="cuda")
    nk.nk_metropolis_sweep(st.ctx, st.params, N, M, c["rule"], None if c["rule"] == "local" else st.edges, s, 0,
                           c["n_discard"], c["n_samples"], st.seed, 0, samples, lp, acc, precision=c["precision"])
    return {"samples": samples, "logpsi": lp, "accepted": acc}


def _run_expect(st, c, N, M):
    eloc = nk.nk_local_energy(st.ctx, st.params, N, M, st.ham, st.s, _empty(c["Ns"]), precision=c["precision"])
    stats = nk.nk_stats(st.ctx, eloc, c["Ns"], _empty(3))
    force = nk.nk_force(st.ctx, st.params, N, M, st.s, eloc, torch.empty_like(st.params), precision=c["precision"])
    return {"eloc": eloc, "stats": stats, "force": force}


def _run_qgt(st, c, N, M):
    return {"Sv": nk.nk_qgt_matvec(st.ctx, st.v, torch.empty_like(st.v), 0.01, params=st.params, N=N, M=M, s=st.s,
                                   precision=c["precision"])}


def _run_jac(st, c, N, M):
    dJ = nk.nk_jacobian(st.ctx, st.params, N, M, st.s, True, 0, c["Ns"], _empty(c["Ns"], st.v.numel()),
                        precision=c["precision"])
    return {"dJ": dJ, "Sv": nk.nk_qgt_matvec(st.ctx, st.v, torch.empty_like(st.v), 0.01, dJ=dJ)}


def _run_solve(st, c, N, M):
    delta = torch.empty_like(st.F)
    nk.nk_sr_solve(st.ctx, st.params, N, M, st.s, st.F, delta, solver=c["solver"], diag_shift=0.01,
                   precision=c["precision"])
    return {"delta": delta}


def _step_out(st, c, N):
    """This step's own copies of the parameters and chains, and its outputs."""
    n = c["C"] * c["n_samples"]
    return (st.params.clone(), st.chains.clone(), _empty(nk.SR_STATS_DOUBLES), _empty(n, N, dtype=torch.int8),
            _empty(n))


def _run_step(st, c, N, M):
    params, s, stats, samples, eloc = _step_out(st, c, N)
    cfg = nk.make_cfg(c["rule"], c["precision"], c["solver"], c["n_discard"], c["n_samples"], 0.01, 0.01, st.seed,
                      cg_tol=1e-6 if c["precision"] == "mixed" else 1e-10)
    nk.nk_sr_step(st.ctx, params, N, M, st.ham, nk.make_chains(s), cfg, stats, samples, eloc)
    return {"params": params, "chains": s, "stats": stats, "samples": samples, "eloc": eloc}


def _run_symm(st, c, N, M):
    params, s, stats, samples, eloc = _step_out(st, c, N)
    cfg = nk.make_cfg(c["rule"], c["precision"], "cholesky", c["n_discard"], c["n_samples"], 0.01, 0.01, st.seed)
    nk.nk_symm_sr_step(st.ctx, params, N, c["alpha"], st.perms, st.ham, nk.make_chains(s), cfg, stats, samples, eloc)
    return {"params": params, "chains": s, "stats": stats, "samples": samples, "eloc": eloc}


def _run_tdvp(st, c, N, M):
    params, s = st.params.clone(), st.chains.clone()
    stats, slope = _empty(len(nk.TDVP_STATS_FIELDS)), torch.empty_like(params)
    cfg = nk.make_tdvp_cfg(c["rule"], c["integrator"], c["real_time"], c["solver"], c["n_discard"], c["n_samples"],
                           0.01, 0.0 if c["solver"] == "svd" else 0.01, st.seed,
                           rcond=1e-12 if c["solver"] == "svd" else 0.0)
    nk.nk_tdvp_step(st.ctx, params, N, M, st.ham, nk.make_chains(s), cfg, stats, slope)
    return {"params": params, "chains": s, "stats": stats, "slope": slope}


def _run_crbm(st, c, N, M):
    n = c["Ns"]
    out = {"logpsi": _empty(n, dtype=torch.complex128), "eloc": _empty(n, dtype=torch.complex128),
           "O": _empty(n, st.params.numel(), dtype=torch.complex128)}
    nk.nk_crbm_logpsi(st.ctx, st.params, N, M, st.s, out["logpsi"])
    nk.nk_crbm_local_energy(st.ctx, st.params, N, M, st.ham, st.s, out["eloc"])
    nk.nk_crbm_jacobian(st.ctx, st.params, N, M, st.s, out["O"])
    return out


# ------------------------------------------------------------------- work ---

def work(case):
    """Bytes: parameters, configurations and vectors in, results out.  Flops:
    2 per hidden unit and site of an activation, 2 per hidden unit of an
    amplitude ratio, 2 per entry of the Jacobian in a product with it, and the
    leading terms of the dense factorisations."""
    op, N, M = case["op"], _sites(case), _hidden(case)
    E = len(_ham(case)["edges"])
    conn = N if "tfim" in case["model"] else E / 2
    Np = N + M + N * M
    if op == "symm":
        Np, M = 1 + case["alpha"] * (1 + N), case["alpha"] * N
    word = 16 if op in ("tdvp", "crbm") else 8
    cplx = 4 if word == 16 else 1  # real products in a complex one
    nbytes = float(word * Np)
    if op == "grad":
        n = case["B"]
        return dict(bytes=nbytes * 2 + n * (N + 16), flops=4.0 * n * N * M)
    if op == "expect":
        n = case["Ns"]
        return dict(bytes=nbytes * 2 + n * (N + 8), flops=4.0 * n * N * M + 2.0 * n * conn * M)
    if op == "qgt":
        n = case["Ns"]
        return dict(bytes=nbytes * 3 + n * N, flops=6.0 * n * N * M)
    if op == "jac":
        n = case["Ns"]
        return dict(bytes=nbytes * 3 + n * N + 8.0 * n * Np, flops=2.0 * n * N * M + 6.0 * n * Np)
    if op == "crbm":
        n = case["Ns"]
        return dict(bytes=nbytes + n * (N + 32) + 16.0 * n * Np, flops=2.0 * cplx * n * (N * M + conn * M))
    if op == "solve":
        n = case["Ns"]
        return dict(bytes=nbytes * 3 + n * N, flops=_solve_flops(case["solver"], n, N, M, Np))
    if op == "sweep":
        sweeps = case["C"] * (case["n_discard"] + case["n_samples"])
        return dict(bytes=nbytes + case["C"] * (N * (1 + case["n_samples"]) + 8 * case["n_samples"] + 8.0),
                    flops=4.0 * sweeps * N * M)
    n = case["C"] * case["n_samples"]
    sweeps = case["C"] * (case["n_discard"] + case["n_samples"])
    flops = 4.0 * cplx * sweeps * N * M + 2.0 * cplx * n * conn * M + 2.0 * n * Np
    if op == "step":
        flops += _solve_flops(case["solver"], n, N, M, Np)
    elif op == "symm":
        flops += float(n) * Np * Np + Np ** 3 / 3.0
    else:  # the real embedding of order 2 Np
        slopes = 2 if case["integrator"] == "heun" else 1
        flops = slopes * (flops + 4.0 * n * Np * Np + (2.0 * Np) ** 3 / 3.0)
    return dict(bytes=nbytes * 2 + case["C"] * N * 2.0 + n * (N + 8.0), flops=flops)


def _solve_flops(solver, n, N, M, Np):
    if solver == "cholesky":
        return float(n) * Np * Np + Np ** 3 / 3.0
    if solver == "cg":  # some 40 products at the start of a run
        return 40 * 4.0 * n * N * M
    return float(n) * n * (N + M) + n ** 3 / 3.0 + 4.0 * n * N * M


# ---------------------------------------------- the same in plain 64 bits ---

def _parts(p, N, M):
    return p[:N], p[N:N + M], p[N + M:].reshape(M, N)


def _lncosh(x):
    y = torch.where(x.real >= 0, x, -x)
    if not torch.is_complex(x):
        return y + torch.log1p(torch.exp(-2.0 * y)) - math.log(2.0)
    w = torch.exp(-2.0 * y)
    re = 0.5 * torch.log1p(2.0 * w.real + w.abs() ** 2)
    return y + torch.complex(re, torch.atan2(w.imag, 1.0 + w.real)) - math.log(2.0)


def _exact_eloc(case, p, s, N, M):
    """Local energies by moving the activations over every connected
    configuration."""
    a, _b, W = _parts(p, N, M)
    sd = s.to(p.dtype)
    th = _b + sd @ W.T
    ham = _ham(case)
    edges = torch.from_numpy(ham["edges"]).long().cuda()
    e1 = len(edges) - ham.get("n_edges2", 0)
    J = torch.full((len(edges),), float(ham["J"]), dtype=torch.float64, device="cuda")
    J[e1:] = float(ham.get("J2", 0.0))
    sr = s.double()
    out = ((sr[:, edges[:, 0]] * sr[:, edges[:, 1]]) @ J).to(p.dtype)
    base = _lncosh(th).sum(1)
    if ham["kind"] == "tfim":
        for i in range(N):
            d = _lncosh(th - 2.0 * sd[:, i:i + 1] * W[:, i]).sum(1) - base - 2.0 * a[i] * sd[:, i]
            out -= float(ham["h"]) * torch.exp(d)
        return out
    for q, (i, k) in enumerate(ham["edges"].tolist()):
        rows = (s[:, i] != s[:, k]).nonzero()[:, 0]
        si = sd[rows, i]
        d = (_lncosh(th[rows] - 2.0 * si[:, None] * (W[:, i] - W[:, k])).sum(1) - base[rows]
             - 2.0 * si * (a[i] - a[k]))
        el = 2.0 * float(J[q])
        if q < e1 and ham["marshall"]:
            el = -el
        out[rows] += el * torch.exp(d)
    return out


def _jtg(T, sd, g):
    """J^T g from tanh(theta) and the configurations."""
    Tg = T * g[:, None]
    return torch.cat([sd.T @ g, Tg.sum(0), (Tg.T @ sd).reshape(-1)])


def _jv(T, sd, v, N, M):
    a, b, W = _parts(v, N, M)
    return sd @ a + T @ b + (T * (sd @ W.T)).sum(1)


def exact(case, seed):
    op = case["op"]
    if op not in ("grad", "expect", "qgt", "jac", "solve", "crbm"):
        return None  # the samples come from the library's own random streams
    N, M = _sites(case), _hidden(case)
    st = prepare(case, seed)
    p, s = st.params, st.s
    a, b, W = _parts(p, N, M)
    sd = s.to(p.dtype)
    th = b + sd @ W.T
    if op == "grad":
        return {"logpsi": sd @ a + _lncosh(th).sum(1), "grad": _jtg(torch.tanh(th), sd, st.g)}
    if op == "crbm":
        T = torch.tanh(th)
        O = torch.cat([sd, T, (T[:, :, None] * sd[:, None, :]).reshape(len(s), -1)], 1)
        return {"logpsi": sd @ a + _lncosh(th).sum(1), "eloc": _exact_eloc(case, p, s, N, M), "O": O}
    T = torch.tanh(th)
    n = len(s)
    if op == "expect":
        e = _exact_eloc(case, p, s, N, M)
        var = ((e - e.mean()) ** 2).mean()
        force = _jtg(T, sd, 2.0 * (e - e.mean()) / n)
        return {"eloc": e, "stats": torch.stack([e.mean(), var, (var / n).sqrt()]), "force": force}
    if op == "qgt":
        w = _jv(T, sd, st.v, N, M) / n
        return {"Sv": _jtg(T, sd, w - w.mean()) + 0.01 * st.v}
    if op == "jac":
        J = torch.cat([sd, T, (T[:, :, None] * sd[:, None, :]).reshape(n, -1)], 1)
        J -= J.mean(0)
        return {"dJ": J, "Sv": J.T @ (J @ st.v) / n + 0.01 * st.v}
    # delta = (F - X^T (X X^T + eps)^-1 X F) / eps, X = dJ / sqrt(n)
    K = (sd @ sd.T + 1.0) * (T @ T.T + 1.0) - 1.0
    K = (K - K.mean(0) - K.mean(1)[:, None] + K.mean()) / n
    K += 0.01 * torch.eye(n, dtype=K.dtype, device="cuda")
    x = _jv(T, sd, st.F, N, M) / math.sqrt(n)
    y = torch.cholesky_solve((x - x.mean())[:, None], torch.linalg.cholesky(K))[:, 0]
    return {"delta": (st.F - _jtg(T, sd, (y - y.mean()) / math.sqrt(n))) / 0.01}
