"""Timed cases of the VMC library: what a user of `paper_1711_11418_gb300.vmc` has it do.

Every case makes its calls through `vmc.Context`.  A case is one of these kinds:

  step      sample, then one SR step on the samples (an optimisation step in FP64)
  sample    Metropolis sweeps with measurements (Sec. 3.1-3.3), energies and configurations out
  gradient  new parameters in (every inverse rebuilt), energies and SR force of given
            configurations out, as an outer optimiser or a line search asks for
  sr        one SR step on given samples (Sec. 3.3.1-3.3.2)
  corr      pair correlations of given configurations (measurement mode, Sec. 2.2.3)
  lanczos   first-step power-Lanczos moments of given configurations (Sec. 3.4)
  project   sampling of a momentum-projected state (Sec. 3.2.2)
  spin      one step of a J1-J2 model: parameters in, exchange sampling, one SR-CG step
  batch     one step of many uneven systems: parameters in, sampling, SR of every system

Results of the mixed form come back in the type its kernels form them in (FP32 ratios, samples
and overlap products), those of the plain form in FP64; configurations and counters are whole.
"""
import functools
import math

import numpy as np
import torch

from paper_1711_11418_gb300 import inputs, vmc

FILL = 0.4375                       # electrons of one spin per site: n = 0.875


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest workload: an 8-site ring, plain FP64, launches and latency count
        dict(name="ring8_step_f64", kind="step", Lx=8, Ly=1, N=4, U=4.0, walkers=64, samples=20,
             sweeps=10, mixed=False),
        # the 8x8 lattice at half filling, plain FP64: an ordinary optimisation step
        dict(name="square8_step_f64", kind="step", Lx=8, Ly=8, N=32, U=4.0, walkers=1024, samples=4,
             sweeps=1, mixed=False),
        # the 16x16 Hubbard workload, mixed form: the sampling half of its optimisation step
        dict(name="hub16_sample_mixed", kind="sample", Lx=16, Ly=16, N=112, U=8.0, walkers=4096,
             samples=4, sweeps=1, mixed=True),
        # the same in the plain FP64 form, fewer walkers
        dict(name="hub16_sample_f64", kind="sample", Lx=16, Ly=16, N=112, U=8.0, walkers=1024,
             samples=1, sweeps=1, mixed=False),
        # energies and force at new parameters: every walker's inverse from scratch
        dict(name="hub16_gradient_mixed", kind="gradient", Lx=16, Ly=16, N=112, U=8.0, walkers=4096,
             mixed=True),
        # the SR half of the 16x16 step: 4096 walkers x 4 samples, 1069 parameters
        dict(name="hub16_sr_mixed", kind="sr", Lx=16, Ly=16, rows=16384, mixed=True),
        # the same solved in the plain form (FP64 S, FP64 Cholesky)
        dict(name="hub16_sr_f64", kind="sr", Lx=16, Ly=16, rows=16384, mixed=False),
        # physical quantities of the 16x16 workload: all site pairs of six kinds
        dict(name="hub16_corr_mixed", kind="corr", Lx=16, Ly=16, N=112, U=8.0, walkers=4096, mixed=True),
        # power-Lanczos moments on the 16x16 workload
        dict(name="hub16_lanczos_mixed", kind="lanczos", Lx=16, Ly=16, N=112, U=8.0, walkers=1024,
             mixed=True),
        # momentum projection with all 256 translations: inverses streamed from memory; three
        # sweeps to a sample, after which most walkers' inverses are due to be rebuilt
        dict(name="hub16_project_mixed", kind="project", Lx=16, Ly=16, N=112, U=8.0, walkers=608,
             sweeps=3, mixed=True),
        # the 16x16 J1-J2 model without symmetry reduction: 65,536 parameters, SR-CG
        dict(name="j1j2_step_mixed", kind="spin", L=16, J2=0.5, walkers=1024, samples=4, batch=8,
             cg=16, mixed=True),
        # 64 independent Hubbard systems of uneven size in one context
        dict(name="batch64_step_mixed", kind="batch", systems=64, walkers=64, samples=4, mixed=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice(rng, lo, hi):
    """Lx <= Ly, odd and rectangular ones among them, with a closed shell near n = 0.6 .. 1."""
    while True:
        Lx, Ly = sorted((rng.randint(lo, hi), rng.randint(lo, hi)))
        N = _closed(Lx, Ly, rng.uniform(0.3, 0.5))
        if N is not None and 2 <= N <= 128:
            return dict(Lx=Lx, Ly=Ly, N=N)


def draw(rng):
    kind = rng.choice(["step", "sample", "sample", "gradient", "sr", "sr", "corr", "lanczos",
                       "project", "spin", "batch"])
    mixed = rng.random() < 0.6
    U = rng.choice([2.0, 4.0, 6.0, 8.0])
    if kind == "step":
        return dict(kind=kind, U=U, walkers=_log(rng, 64, 1024), samples=rng.randint(1, 8),
                    sweeps=rng.randint(1, 4), mixed=False, **_lattice(rng, 3, 8))
    if kind == "sample":
        return dict(kind=kind, U=U, walkers=_log(rng, 64, 4096 if mixed else 1024),
                    samples=rng.randint(1, 4) if mixed else 1, sweeps=1, mixed=mixed,
                    **_lattice(rng, 4, 16))
    if kind == "gradient":
        return dict(kind=kind, U=U, walkers=_log(rng, 64, 4096), mixed=mixed, **_lattice(rng, 4, 16))
    if kind == "sr":
        Lx, Ly = sorted((rng.randint(4, 16), rng.randint(4, 16)))
        return dict(kind=kind, Lx=Lx, Ly=Ly, rows=_log(rng, 256, 16384), mixed=mixed)
    if kind == "corr":
        return dict(kind=kind, U=U, walkers=_log(rng, 64, 4096 if mixed else 256), mixed=mixed,
                    **_lattice(rng, 4, 16))
    if kind == "lanczos":
        return dict(kind=kind, U=U, walkers=_log(rng, 64, 1024 if mixed else 64), mixed=mixed,
                    **_lattice(rng, 4, 16))
    if kind == "project":
        lat = _lattice(rng, 4, 8)
        return dict(kind=kind, U=U, walkers=_log(rng, 64, 608), sweeps=3, mixed=mixed, **lat)
    if kind == "spin":
        return dict(kind=kind, L=2 * rng.randint(2, 7), J2=rng.choice([0.0, 0.25, 0.5]),
                    walkers=_log(rng, 64, 1024), samples=rng.randint(1, 4), batch=rng.choice([1, 2, 4, 8]),
                    cg=16, mixed=True)
    return dict(kind="batch", systems=rng.randint(2, 48), walkers=_log(rng, 16, 64),
                samples=rng.randint(1, 4), mixed=True)


# --------------------------------------------------------------------------- inputs
def _levels(Lx, Ly, bx, by):
    k = lambda L, b: 2 * np.pi * np.arange(L) / L + (0.0 if b == 1 else np.pi / L)  # noqa: E731
    return np.sort((-2 * np.cos(k(Lx, bx))[:, None] - 2 * np.cos(k(Ly, by))[None, :]).ravel())


BOUNDS = ((-1, -1), (1, -1), (-1, 1), (1, 1))


def _shell(Lx, Ly, N):
    """Boundary signs that close the shell at N, or None."""
    for bx, by in BOUNDS:
        e = _levels(Lx, Ly, bx, by)
        if N < e.size and e[N] - e[N - 1] > 1e-6:
            return bx, by
    return None


def _closed(Lx, Ly, fill):
    want = fill * Lx * Ly
    for N in sorted(range(2, Lx * Ly // 2 + 1), key=lambda n: abs(n - want)):
        if _shell(Lx, Ly, N):
            return N
    return None


@functools.lru_cache(maxsize=32)
def _base(Lx, Ly, N, U):
    if Ly == 1:
        return inputs.ring8_hubbard(noise=0.0, U=U)
    bx, by = _shell(Lx, Ly, N) if (Lx, Ly, N) != (8, 8, 32) else (1, -1)
    sub = (2 if Lx % 2 == 0 else 1, 2 if Ly % 2 == 0 else 1)
    return inputs.make_problem("hubbard", inputs.square(Lx, Ly, bx, by), 2 * N, U=U, sub=sub,
                               jastrow="distance", noise=0.0)


def _problem(case, seed):
    """The Hubbard problem with the U = 0 pairing plus noise, and correlation factors as an
    optimised state has them: doublons suppressed, a Jastrow factor that falls off."""
    p = _base(case["Lx"], case["Ly"], case["N"], case["U"])
    rng = np.random.default_rng(seed)
    a = p.params.copy()
    a[:p.n_g] = -0.1 * case["U"] * rng.uniform(0.8, 1.2)
    a[p.n_g:p.n_g + p.n_v] = 0.15 * rng.uniform(0.5, 1.0, p.n_v) / (1.0 + np.arange(p.n_v))
    a[p.n_g + p.n_v:] += rng.uniform(-0.05, 0.05, p.n_f)
    return p.copy_with(params=a)


def _slater(Phi, W, gen):
    """W sets of N sites drawn from det^2 of the orbitals Phi [Ns, N] (one spin of the U = 0
    state, where the pairing state is a Slater determinant): sites one at a time, each with the
    weight left to it by those already taken."""
    Ns, N = Phi.shape
    V = torch.as_tensor(Phi, device="cuda")
    left = (V * V).sum(1).expand(W, Ns).clone()
    Q = torch.zeros(W, N, N, dtype=torch.float64, device="cuda")
    out = torch.empty(W, N, dtype=torch.int64, device="cuda")
    ar = torch.arange(W, device="cuda")
    for k in range(N):
        u = torch.rand(W, Ns, generator=gen, device="cuda", dtype=torch.float64)
        pick = (left.clamp_min(1e-14).log() - (-u.clamp_min(1e-300).log()).log()).argmax(1)
        out[:, k] = pick
        v = V[pick]
        for _ in range(2):
            v = v - torch.bmm(torch.bmm(v[:, None, :], Q[:, :k].transpose(1, 2)), Q[:, :k])[:, 0]
        v = v / v.norm(dim=1, keepdim=True).clamp_min(1e-150)
        Q[:, k] = v
        left = (left - (v @ V.T) ** 2).clamp_min(0.0)
        left.scatter_(1, out[:, :k + 1], 0.0)
    return out


@functools.lru_cache(maxsize=32)
def _orbitals(Lx, Ly, N, U):
    p = _base(Lx, Ly, N, U)
    return inputs.free_fermion_orbitals(p.lat, (p.hop_i, p.hop_j, p.hop_t), N)


def _configs(case, seed, W):
    """[W, 2N] electron placements in label order: the up and down electrons of the U = 0 state."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    Phi = _orbitals(case["Lx"], case["Ly"], case["N"], case["U"])
    n = min(W, 1024)
    up, dn = _slater(Phi, n, gen), _slater(Phi, n, gen)
    cpu = torch.Generator().manual_seed(seed + 1)
    iu = torch.cat([torch.randperm(n, generator=cpu) for _ in range(-(-W // n))])[:W]
    idn = torch.cat([torch.randperm(n, generator=cpu) for _ in range(-(-W // n))])[:W]
    return torch.cat([up.cpu()[iu], dn.cpu()[idn]], 1).to(torch.int32).numpy()


def _sr_problem(case):
    Lx, Ly = case["Lx"], case["Ly"]
    return _base(Lx, Ly, _closed(Lx, Ly, FILL), 8.0)


def _sr_samples(rows, Np, seed):
    """(E, O): correlated columns of uneven size, as sampled log-derivatives are."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.randn(*s, generator=gen, device="cuda")  # noqa: E731
    size = torch.exp(0.7 * r(1, Np))
    O = (r(rows, Np) * torch.exp(0.4 * r(rows, 1)) + r(rows, 16) @ r(16, Np) * 0.25) * size + 0.3 * r(1, Np)
    E = -100.0 + 3.0 * r(rows).double() + (O[:, :min(Np, 24)] / size[:, :min(Np, 24)]).double().sum(1) * 0.3
    return E.cpu().numpy(), O.cpu().numpy()


def _precision(case):
    return vmc.MIXED if case["mixed"] else vmc.FP64


def prepare(case, seed):
    kind, W = case["kind"], case.get("walkers")
    if kind == "sr":
        p, rows = _sr_problem(case), case["rows"]
        ctx = vmc.Context(p, -(-rows // 4), seed=seed, precision=_precision(case), max_samples=4)
        E, O = _sr_samples(rows, p.Np, seed)
        ctx.set_samples(E, O)
        return dict(case=case, ctx=ctx)
    if kind == "spin":
        p = inputs.j1j2_heisenberg(case["L"], J2=case["J2"], seed=seed)
        ctx = vmc.Context(p, W, seed=seed, precision=_precision(case), max_samples=case["samples"])
        ctx.set_proposal_batch(case["batch"])
        ctx.sample(4, 0, 0)
        return dict(case=case, ctx=ctx, params=p.params)
    if kind == "batch":
        probs = _batch(case["systems"])
        rng = np.random.default_rng(seed)
        probs = [p.copy_with(params=p.params * rng.uniform(0.95, 1.05, p.params.size)) for p in probs]
        ctx = vmc.Context(probs, W, seed=seed, precision=_precision(case), max_samples=case["samples"],
                          recompute_every=64)
        ctx.sample(4, 0, 0)
        return dict(case=case, ctx=ctx, params=[p.params for p in probs])
    p = _problem(case, seed)
    ctx = vmc.Context(p, W, seed=seed, precision=_precision(case), max_samples=case.get("samples", 1))
    ctx.set_configs(_configs(case, seed, W) if case["Ly"] > 1 else
                    inputs.initial_configs(p.Ns, p.Ne, W, False, seed))
    if kind == "project":
        perm, sign = inputs.translation_ops(p.lat)
        ctx.set_projection(perm, sign, np.full(len(perm), 1.0 / len(perm)))
    ctx.sample(0, 0, 0)             # the inverses of these configurations
    return dict(case=case, ctx=ctx, params=p.params)


@functools.lru_cache(maxsize=8)
def _batch(systems):
    return inputs.batched_hubbard(systems)


# --------------------------------------------------------------------------- one pass
def _t(x, mixed):
    return np.asarray(x, np.float32) if mixed else np.asarray(x, np.float64)


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind, mixed = case["kind"], case["mixed"]
    if kind == "step":
        ctx.sample(0, case["samples"], case["sweeps"])
        E, _ = ctx.get_samples(with_O=False)
        ctx.sr_step(0.02, 1e-3, 1e-4, solver=vmc.CHOLESKY)
        ele, ctr = ctx.get_configs()
        return dict(E=_t(E, mixed), params=_t(ctx.get_params(), mixed), ele=ele, ctr=ctr.astype(np.int64))
    if kind in ("sample", "project"):
        ctx.sample(0, case.get("samples", 1), case.get("sweeps", 1))
        E, _ = ctx.get_samples(with_O=False)
        ele, ctr = ctx.get_configs()
        return dict(E=_t(E, mixed), ele=ele, ctr=ctr.astype(np.int64))
    if kind == "gradient":
        ctx.set_params(state["params"])
        ctx.sample(0, 1, 0)
        E, _ = ctx.get_samples(with_O=False)
        _, g = ctx.get_sr_matrices(with_S=False)
        return dict(E=_t(E, mixed), g=_t(g, mixed))
    if kind == "sr":
        r = ctx.sr_step(0.05, 1e-3, 0.0, solver=vmc.MIXED_IR if mixed else vmc.CHOLESKY, cg_eps=1e-12)
        return dict(params=_t(ctx.get_params(), mixed), energy=_t(r["energy"], mixed),
                    norm_g=_t(r["norm_g"], mixed))
    if kind == "corr":
        return _t(ctx.measure_corr(), mixed)
    if kind == "lanczos":
        F1, F2, h = ctx.lanczos_moments()
        return dict(F1=_t(F1, mixed), F2=_t(F2, mixed), h=_t([h[k] for k in sorted(h)], mixed))
    if kind == "spin":
        ctx.set_params(state["params"])
        ctx.sample(0, case["samples"], 1)
        E, _ = ctx.get_samples(with_O=False)
        ctx.sr_step(0.02, 1e-3, 1e-3, solver=vmc.CG, cg_eps=1e-6, cg_kmax=case["cg"])
        ele, ctr = ctx.get_configs()
        return dict(E=_t(E, mixed), params=_t(ctx.get_params(), mixed), ele=ele, ctr=ctr.astype(np.int64))
    # batch
    n = len(ctx.problems)
    for s in range(n):
        ctx.set_params(state["params"][s], s)
    ctx.sample(0, case["samples"], 1)
    E = np.concatenate([ctx.get_samples(s, with_O=False)[0] for s in range(n)])
    ctx.sr_step_all(0.02, 1e-3, 1e-3, solver=vmc.MIXED_IR, cg_eps=1e-12)
    conf = [ctx.get_configs(s) for s in range(n)]
    return dict(E=_t(E, mixed), params=_t(np.concatenate([ctx.get_params(s) for s in range(n)]), mixed),
                ele=np.concatenate([c[0].ravel() for c in conf]),
                ctr=np.concatenate([c[1] for c in conf]).astype(np.int64))


# --------------------------------------------------------------------------- work
def _sweep_work(Ns, N, W, sweeps, samples, p_ex, Np, es, terms, hold):
    """(bytes, flops) of W walkers' sweeps and measurements: the state in and out once, the
    sample rows out; a tested hop 2N, a tested exchange 2N^2, an accepted move (12 %) 4N^2, a
    measured hop ratio 2N."""
    rho = N / Ns
    props = 2 * N * sweeps
    tested_h, tested_x = props * (1 - p_ex) * (1 - rho), props * p_ex * (1 - rho) ** 2
    fl = W * (tested_h * 2 * N + tested_x * 2 * N * N + 0.12 * props * 4 * N * N
              + samples * terms * 2 * rho * (1 - rho) * 2 * N)
    by = W * (2 * hold * N * N + 2 * 4 * (2 * N + 2 * Ns) + samples * (8 + es * Np))
    return by, fl


def _sr_work(rows, Np, es):
    return es * rows * Np + 8 * rows + 24 * Np, float(rows) * Np * (Np + 1) + Np ** 3 / 3.0


def work(case):
    kind, mixed = case["kind"], case["mixed"]
    es, hold = (4, 8) if mixed else (8, 8)
    if kind == "sr":
        b, f = _sr_work(case["rows"], _sr_problem(case).Np, es)
        return dict(bytes=b, flops=f)
    W = case["walkers"]
    if kind == "spin":
        Ns = case["L"] ** 2
        N, nb, rows = Ns // 2, (4 if case["J2"] else 2) * Ns, W * case["samples"]
        b, f = _sweep_work(Ns, N, W, case["samples"], 0, 0.0, Ns * Ns, es, 0, hold)
        f += W * (2.0 * N ** 3 + case["samples"] * (Ns * 0.5 * 2 * N * N + 2 * N * 2.0 * N * N / 2 + nb * 8 * N))
        return dict(bytes=b + (1 + 2 * case["cg"]) * es * rows * Ns * Ns, flops=f + case["cg"] * 4.0 * rows * Ns * Ns)
    if kind == "batch":
        b = f = 0.0
        for p in _batch(case["systems"]):
            s = _sweep_work(p.Ns, p.N, W, case["samples"], case["samples"], p.p_exchange, p.Np, es,
                            p.hop_i.size, hold)
            r = _sr_work(W * case["samples"], p.Np, es)
            b, f = b + s[0] + r[0], f + s[1] + r[1] + W * 2.0 * p.N ** 3
        return dict(bytes=b, flops=f)
    p = _base(case["Lx"], case["Ly"], case["N"], case["U"])
    N, Ns = p.N, p.Ns
    if kind in ("step", "sample"):
        k = case["samples"]
        b, f = _sweep_work(Ns, N, W, k * case["sweeps"], k, p.p_exchange, p.Np, es, p.hop_i.size, hold)
        if kind == "step":
            r = _sr_work(W * k, p.Np, es)
            b, f = b + r[0], f + r[1] + W * 2.0 * N ** 3
        return dict(bytes=b, flops=f)
    if kind == "gradient":
        b, f = _sweep_work(Ns, N, W, 0, 1, 0.0, p.Np, es, p.hop_i.size, hold)
        return dict(bytes=b + es * W * p.Np, flops=f + W * 2.0 * N ** 3)
    if kind == "corr":
        return dict(bytes=W * (es * N * N + 4 * 4 * Ns) + 48 * Ns * Ns, flops=W * 6.0 * Ns * N * N)
    if kind == "lanczos":
        rho = N / Ns
        pairs = (2 * p.hop_i.size * rho * (1 - rho)) ** 2
        return dict(bytes=W * (es * N * N + 4 * 4 * Ns + 16),
                    flops=W * (2.0 * (2 * Ns * N * N + Ns * Ns * N) + 12 * pairs))
    # project: one inverse per translation, what the fast updates of the sweeps move (12 % accepted)
    rho, props, px = N / Ns, 2 * N * case["sweeps"], p.p_exchange
    th, tx = props * (1 - px) * (1 - rho), props * px * (1 - rho) ** 2
    words = th * N + tx * N * N + 0.12 * props * 3 * N * N + N * N
    return dict(bytes=es * W * Ns * words, flops=2.0 * W * Ns * words)


# --------------------------------------------------------------------------- 64-bit values
def _tables(f, ele, N):
    """(M^-1, G_up[w, b, k], G_dn[w, a, m], T[w, b, a]) of configurations ele [w, 2N]."""
    up, dn = ele[:, :N], ele[:, N:]
    B = torch.linalg.inv(f[up[:, :, None], dn[:, None, :]])
    Gu = f[:, dn].permute(1, 0, 2) @ B
    Gd = f.T[:, up].permute(1, 0, 2) @ B.transpose(1, 2)
    return B, Gu, Gd, Gu @ f[up]


def _exact_inputs(case, seed):
    p = _problem(case, seed)
    dev = dict(device="cuda", dtype=torch.float64)
    f = torch.as_tensor(p.f_matrix(), **dev)
    ele = torch.as_tensor(_configs(case, seed, case["walkers"]), device="cuda").long()
    vi = torch.as_tensor(p.v_idx, device="cuda").long().reshape(p.Ns, p.Ns)
    v = torch.where(vi >= 0, torch.as_tensor(p.params[p.n_g:p.n_g + p.n_v], **dev)[vi.clamp_min(0)], 0.0)
    g = float(p.params[0])
    return p, f, v, g, ele


def _state(p, v, ele):
    """Occupations of both spins and the Jastrow field of configurations."""
    w, N = ele.shape[0], p.N
    nu = torch.zeros(w, p.Ns, device="cuda", dtype=torch.float64).scatter_(1, ele[:, :N], 1.0)
    nd = torch.zeros(w, p.Ns, device="cuda", dtype=torch.float64).scatter_(1, ele[:, N:], 1.0)
    return nu, nd, (nu + nd - 1.0) @ v


def _by_site(G, lab, Ns):
    """Columns by electron label -> columns by site (0 at empty ones)."""
    return torch.zeros(G.shape[0], G.shape[1], Ns, device="cuda", dtype=torch.float64).scatter_(
        2, lab[:, None, :].expand(-1, G.shape[1], -1), G)


def _hops(p, v, g, nu, nd, h, GU, GD):
    """Per term and spin: psi(x')/psi(x) of the hop j -> i (0 where there is none)."""
    i, j = (torch.as_tensor(a, device="cuda").long() for a in (p.hop_i, p.hop_j))
    dj = h[:, i] - h[:, j] - v[j, i]
    ru = GU[:, i, j] * torch.exp(dj + g * (nd[:, i] - nd[:, j])) * nu[:, j] * (1 - nu[:, i])
    rd = GD[:, i, j] * torch.exp(dj + g * (nu[:, i] - nu[:, j])) * nd[:, j] * (1 - nd[:, i])
    return ru, rd


def _exact_gradient(case, seed):
    p, f, v, g, ele = _exact_inputs(case, seed)
    N, W = p.N, case["walkers"]
    t = torch.as_tensor(p.hop_t, device="cuda", dtype=torch.float64)
    fi = torch.as_tensor(p.f_idx, device="cuda").long().reshape(p.Ns, p.Ns)
    fs = torch.as_tensor(p.f_sign, device="cuda").double().reshape(p.Ns, p.Ns)
    vi = torch.as_tensor(p.v_idx, device="cuda").long().reshape(-1)
    E, O = [], []
    for e in ele.split(256):
        B, Gu, Gd, _ = _tables(f, e, N)
        nu, nd, h = _state(p, v, e)
        ru, rd = _hops(p, v, g, nu, nd, h, _by_site(Gu, e[:, :N], p.Ns), _by_site(Gd, e[:, N:], p.Ns))
        D = (nu * nd).sum(1)
        E.append(case["U"] * D - ((ru + rd) * t).sum(1))
        m = nu + nd - 1.0
        o = torch.zeros(len(e), p.Np, device="cuda", dtype=torch.float64)
        o[:, 0] = D
        mm = (m[:, :, None] * m[:, None, :]).reshape(len(e), -1)
        ok = vi >= 0
        o.index_add_(1, p.n_g + vi[ok], 0.5 * mm[:, ok])
        up, dn = e[:, :N], e[:, N:]
        c = fi[up[:, :, None], dn[:, None, :]]
        o.scatter_add_(1, (p.n_g + p.n_v + c).reshape(len(e), -1),
                       (B.transpose(1, 2) * fs[up[:, :, None], dn[:, None, :]]).reshape(len(e), -1))
        O.append(o)
    E, O = torch.cat(E), torch.cat(O)
    return dict(E=E, g=(O - O.mean(0)).T @ (E - E.mean()) / W)


def _exact_sr(case, seed):
    p, rows = _sr_problem(case), case["rows"]
    E, O = (torch.as_tensor(a, device="cuda").double() for a in _sr_samples(rows, p.Np, seed))
    X, e = O - O.mean(0), E - E.mean()
    g = X.T @ e / rows
    S = X.T @ X / rows
    S += torch.diag(S.diagonal() * 1e-3)
    x = torch.linalg.solve(S, g)
    r = g - S @ x
    x = x + torch.linalg.solve(S, r)
    return dict(params=torch.as_tensor(p.params, device="cuda") - 0.05 * x, energy=E.mean(), norm_g=g.norm())


def _exact_corr(case, seed):
    p, f, v, g, ele = _exact_inputs(case, seed)
    N, Ns = p.N, p.Ns
    out = torch.zeros(6, Ns, Ns, device="cuda", dtype=torch.float64)
    off = 1.0 - torch.eye(Ns, device="cuda", dtype=torch.float64)
    for e in ele.split(256):
        B, Gu, Gd, T = _tables(f, e, N)
        nu, nd, h = _state(p, v, e)
        GU, GD = _by_site(Gu, e[:, :N], Ns), _by_site(Gd, e[:, N:], Ns)
        BS = _by_site(torch.zeros(len(e), Ns, N, device="cuda", dtype=torch.float64).scatter_(
            1, e[:, N:, None].expand(-1, -1, N), B), e[:, :N], Ns)          # [w, down site, up site]
        dj = h[:, :, None] - h[:, None, :] - v
        P = lambda o: torch.exp(dj + g * (o[:, :, None] - o[:, None, :]))  # noqa: E731
        out[0] += (GU * P(nd) * nu[:, None, :] * (1 - nu)[:, :, None]).sum(0) * off
        out[1] += (GD * P(nu) * nd[:, None, :] * (1 - nd)[:, :, None]).sum(0) * off
        n, s = nu + nd, 0.5 * (nu - nd)
        out[2] += n.T @ n
        out[3] += s.T @ s
        b, a = nd * (1 - nu), nu * (1 - nd)                                 # S+ on b, S- on a
        swap = GU * GD.transpose(1, 2) - BS * (T - f)
        out[4] += -(swap * b[:, :, None] * a[:, None, :]).sum(0) * off
        out[0] += torch.diag(nu.sum(0))
        out[1] += torch.diag(nd.sum(0))
        out[4] += torch.diag((nu * (1 - nd)).sum(0))
        out[5] += torch.diag((0.5 * (nu + nd) - nu * nd).sum(0))
    od = out[4] * off
    out[5] += out[3] + 0.5 * (od + od.T)
    return out / case["walkers"]


def _exact_lanczos(case, seed):
    p, f, v, g, ele = _exact_inputs(case, seed)
    N, Ns, U = p.N, p.Ns, case["U"]
    i, j = (torch.as_tensor(a, device="cuda").long() for a in (p.hop_i, p.hop_j))
    t = torch.as_tensor(p.hop_t, device="cuda", dtype=torch.float64)
    I, J, H = i.repeat(2), j.repeat(2), -t.repeat(2)
    s = torch.arange(2, device="cuda").repeat_interleave(i.numel())
    F1, F2 = [], []
    for e in ele.split(128):
        B, Gu, Gd, T = _tables(f, e, N)
        nu, nd, h = _state(p, v, e)
        GU, GD = _by_site(Gu, e[:, :N], Ns), _by_site(Gd, e[:, N:], Ns)
        BS = _by_site(torch.zeros(len(e), Ns, N, device="cuda", dtype=torch.float64).scatter_(
            1, e[:, N:, None].expand(-1, -1, N), B), e[:, :N], Ns)
        R1 = torch.cat(_hops(p, v, g, nu, nd, h, GU, GD), 1)
        D = U * (nu * nd).sum(1)
        E1 = D + R1 @ H
        n2 = torch.stack([nu, nd], 1)
        for w in range(len(e)):
            q = torch.nonzero((n2[w][s, J] > 0) & (n2[w][s, I] == 0))[:, 0]
            o = n2[w]
            G = torch.stack([GU[w], GD[w]])
            s1, i1, j1 = s[q][:, None], I[q][:, None], J[q][:, None]
            S2, I2, J2 = s[None], I[None], J[None]
            # occupations of x' = (j1 -> i1) x
            occ = lambda sp, x: o[sp, x] + (sp == s1) * ((x == i1).double() - (x == j1).double())  # noqa: E731
            ok = (occ(S2, J2) > 0.5) & (occ(S2, I2) < 0.5)
            same = S2 == s1
            again = same & (J2 == i1)
            c1 = h[w][i1] - h[w][j1] - v[j1, i1] + g * (o[1 - s1, i1] - o[1 - s1, j1])
            c2 = (h[w][I2] + v[I2, i1] - v[I2, j1]) - (h[w][J2] + v[J2, i1] - v[J2, j1]) - v[J2, I2]
            c2 = c2 + g * (occ(1 - S2, I2) - occ(1 - S2, J2))
            det_same = G[s1, i1, j1] * G[S2, I2, J2] - G[s1, i1, J2] * G[S2, I2, j1]
            b, ju = torch.where(s1 == 0, i1, I2), torch.where(s1 == 0, j1, J2)
            a, jd = torch.where(s1 == 0, I2, i1), torch.where(s1 == 0, J2, j1)
            det_opp = G[0][b, ju] * G[1][a, jd] - BS[w][jd, ju] * (T[w][b, a] - f[b, a])
            R = torch.where(same, det_same, det_opp) * torch.exp(c1 + c2)
            # the same electron again: one hop j1 -> i2 of x, or back to x
            ca = h[w][I2] - h[w][j1] - v[j1, I2] + g * (o[1 - s1, I2] - o[1 - s1, j1])
            Ra = torch.where(I2 == j1, torch.ones_like(ca), G[s1, I2, j1] * torch.exp(ca))
            R = torch.where(again, Ra, R)
            R = torch.where(ok, R, torch.zeros_like(R))
            dx = D[w] + U * (o[1 - s1, i1] - o[1 - s1, j1])[:, 0]
            F2.append(D[w] * E1[w] + (H[q] * (dx * R1[w][q] + R @ H)).sum())
        F1.append(E1)
    F1, F2 = torch.cat(F1), torch.stack(F2)
    h = dict(h1=F1.mean(), h2_11=(F1 * F1).mean(), h2_20=F2.mean(), h3_12=(F1 * F2).mean())
    return dict(F1=F1, F2=F2, h=torch.stack([h[k] for k in sorted(h)]))


def exact(case, seed):
    """Markov chains (step, sample, project, spin, batch) have no value that goes without the
    library's random stream; the others are determinants, ratios and linear systems."""
    kind = case["kind"]
    v = (_exact_gradient if kind == "gradient" else _exact_sr if kind == "sr" else _exact_corr if kind == "corr"
         else _exact_lanczos if kind == "lanczos" else None)
    if v is None:
        return None
    torch.backends.cuda.matmul.allow_tf32 = False
    return v(case, seed)
