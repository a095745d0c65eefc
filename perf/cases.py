"""The work that this library is measured on: the sampler, its learned screen,
molecular dynamics and the reweighting, each through the calls a user's program
makes, over the range of sizes that the workloads, tests and benchmark of this
repository use.

A case is a dict of plain values.  ``listed()`` gives the fixed ones,
``draw(rng)`` one more of the same ranges; ``prepare`` builds what a program
holds before the call, ``run`` makes one pass, ``work`` states what a pass
cannot do without, and ``exact`` gives the reweighting's results in 64 bits.
"""
import math

import numpy as np
import torch

import workloads as W
from paper_1908_11118_gb300 import Batch, Regc, mbar_query, mbar_solve


def listed():
    return [
        # the smallest grid in use: 16 replicas on a 4x4x2 slab, a user's shortest
        # interactive step (ten sweeps, one exchange, the walkers read back)
        dict(name="grid_16_fcc100", kind="sweep", system="fcc100", L=4, M=4, nmax=32, sweeps=10, blocks=1),
        # the benchmark's grid: 1024 replicas over the 12x12x4 slab, a stretch of a
        # production run with an exchange every ten sweeps
        dict(name="grid_1024_fcc111", kind="sweep", system="fcc111", L=32, M=32, nmax=512, sweeps=10, blocks=10),
        # the paper's own run: 160 replicas of the LJ A18 system, the x0 cycle with ten
        # displacements a step, a structure sample every 100 steps
        dict(name="cycle_160_a18", kind="cycle", L=10, M=16, nmax=160, steps=100, blocks=4),
        # two reactive gases on a (T, mu_B, mu_C) grid
        dict(name="two_gas_1024", kind="sweep", system="two_gas", L=8, M=16, K=8, nmax=256, sweeps=10, blocks=5),
        # the cluster-in-gas workload: 4096 small walkers in a periodic cube, no surface
        dict(name="cluster_4096", kind="sweep", system="cluster", L=64, M=64, nmax=64, sweeps=10, blocks=5),
        # delayed acceptance with a trained network on the benchmark's grid
        dict(name="delayed_1024_fcc111", kind="sweep", system="fcc111", L=32, M=32, nmax=512, sweeps=10, blocks=3,
             delayed=True),
        # many uneven systems (Nmax 64 .. 2048, ragged slabs) stepped together
        dict(name="batch_64_uneven", kind="batch", systems=64, L=4, M=4, lo=6, hi=11, sweeps=10, blocks=2),
        # REGCMD: particle exchanges with MD segments in between
        dict(name="md_1024_fcc111", kind="md", L=32, M=32, nmax=512, steps=4, md_steps=10),
        # one step with every walker handed in from and back to page-locked host memory,
        # as a driver program that owns the configurations does it
        dict(name="walkers_1024_fcc111", kind="walkers", L=32, M=32, nmax=512, sweeps=10),
        # MBAR over a caller's pooled bins: the paper's 160 states, a 12 x 12 phase map
        dict(name="mbar_160", kind="mbar", L=10, M=16, nmax=100, e_bin=0.25, obs=4000, Q=12),
        # the reweighting of a handle's own histograms after a run on the benchmark's grid
        dict(name="reweight_1024_fcc111", kind="reweight", L=32, M=32, nmax=512, sweeps=2000, Q=12),
        # the learning phase of delayed acceptance: rows harvested along the run, then
        # mini-batch training
        dict(name="train_fcc111", kind="train", L=8, M=8, nmax=512, harvests=8, steps=500, batch=1024),
    ]


def _log_int(rng, lo, hi):
    """A whole number spread over the logarithm of lo .. hi."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["sweep"] * 6 + ["cycle"] * 2 + ["batch", "md", "walkers", "mbar", "mbar", "reweight", "train"])
    if kind == "sweep":
        system = rng.choice(["fcc100", "fcc111", "fcc111", "two_gas", "cluster", "delayed"])
        c = dict(kind="sweep", system="fcc111" if system == "delayed" else system, L=_log_int(rng, 2, 32),
                 M=_log_int(rng, 3, 32), sweeps=rng.randint(5, 20), blocks=rng.randint(1, 5))
        if system == "fcc100":
            c["nmax"] = _log_int(rng, 8, 64)
        elif system == "cluster":
            c.update(L=_log_int(rng, 3, 64), M=_log_int(rng, 3, 64), nmax=_log_int(rng, 16, 96))
        elif system == "two_gas":
            c.update(L=_log_int(rng, 2, 8), M=_log_int(rng, 2, 16), K=_log_int(rng, 2, 8), nmax=_log_int(rng, 24, 256))
        else:
            c["nmax"] = _log_int(rng, 48, 512)
            if system == "delayed":
                c.update(delayed=True, blocks=rng.randint(1, 2))
        return c
    if kind == "cycle":
        return dict(kind=kind, L=_log_int(rng, 2, 10), M=_log_int(rng, 3, 16), nmax=_log_int(rng, 40, 160),
                    steps=rng.randint(30, 150), blocks=rng.randint(1, 3))
    if kind == "batch":
        lo = rng.randint(6, 9)
        return dict(kind=kind, systems=_log_int(rng, 5, 60), L=rng.randint(2, 4), M=rng.randint(2, 4), lo=lo,
                    hi=rng.randint(lo, 11), sweeps=rng.randint(5, 10), blocks=rng.randint(1, 2))
    if kind == "md":
        return dict(kind=kind, L=_log_int(rng, 3, 32), M=_log_int(rng, 3, 32), nmax=_log_int(rng, 48, 512),
                    steps=rng.randint(1, 4), md_steps=rng.randint(3, 10))
    if kind == "walkers":
        return dict(kind=kind, L=_log_int(rng, 3, 32), M=_log_int(rng, 3, 32), nmax=_log_int(rng, 48, 512),
                    sweeps=rng.randint(3, 10))
    if kind == "mbar":
        return dict(kind=kind, L=_log_int(rng, 3, 10), M=_log_int(rng, 4, 16), nmax=_log_int(rng, 20, 100),
                    e_bin=rng.uniform(0.25, 1.0), obs=_log_int(rng, 500, 4000), Q=rng.randint(3, 12))
    if kind == "reweight":
        return dict(kind=kind, L=_log_int(rng, 8, 31), M=_log_int(rng, 8, 31), nmax=_log_int(rng, 64, 512),
                    sweeps=_log_int(rng, 300, 2000), Q=rng.randint(3, 12))
    return dict(kind=kind, L=_log_int(rng, 3, 8), M=_log_int(rng, 3, 8), nmax=_log_int(rng, 48, 512),
                harvests=rng.randint(2, 8), steps=_log_int(rng, 50, 500), batch=_log_int(rng, 100, 1024))


# ---------------------------------------------------------------- preparation

def _pinned(shape, dtype):
    return torch.zeros(shape, dtype=dtype, pin_memory=True).numpy()


def _out(g):
    """Page-locked buffers for a handle's walkers."""
    return (_pinned((g.S, g.nmax, 3), torch.float32), _pinned((g.S,), torch.int32), _pinned((g.S,), torch.float64),
            _pinned((g.S,), torch.int32))


def _problem(c, seed):
    kw = dict(seed=seed % 65521, nmax=c["nmax"], L=c["L"], M=c["M"])
    if c["kind"] == "cycle":
        return W.lj_a18_hex_slab(**kw)
    system = c.get("system", "fcc111")
    if system == "fcc100":
        return W.fcc100_small(**kw)
    if system == "two_gas":
        return W.two_gas_paper_scale(K=c["K"], **kw)
    if system == "cluster":
        return W.cluster_in_gas(L=c["L"], M=c["M"], nmax_b=c["nmax"], seed=kw["seed"])
    return W.fcc111_paper_scale(**kw)


def _walkers(c, p, seed):
    """Starting configurations as a user's run begins: (pos, n, nb or None)."""
    rng = np.random.default_rng(seed)
    if c["kind"] == "cycle":
        return np.zeros((p.S, p.nmax, 3)), np.zeros(p.S, np.int32), None     # the pristine slab
    if p.n_cluster:
        pos, n = W.cluster_initial(p, rng.integers(0, c["nmax"] // 2 + 1, p.S), seed=seed)
        return pos, n, None
    cap = int(0.9 * W.lattice_sites(p))
    pos, n = W.lattice_walkers(p, np.minimum(rng.integers(0, p.nmax // 2 + 1, p.S), cap), seed=seed)
    return pos, n, (n // 2).astype(np.int32) if p.gc2_type else None


def _grid(c, seed, equilibrate=200):
    """A handle that holds walkers of a run under way."""
    p = _problem(c, seed)
    pos, n, nb = _walkers(c, p, seed)
    g = Regc(p)
    g.set_walkers(pos, n, nb=nb)
    if equilibrate:
        g.run(equilibrate, 10)
    return g


def _learn(g, harvests, steps, seed):
    g.surrogate_init(seed % 65521)
    rows = 16 * g.S
    for _ in range(harvests):
        g.sweep(10)
        g.surrogate_harvest(8, 8, 8.0, harvests * rows)
    if steps:
        g.surrogate_train(steps, 1024, 1e-3)


def _bins(c, seed):
    """Pooled (N, E) bins of a run on an L x M grid: every state's observations drawn
    from the grand-canonical law of a gas whose energy at N is Gaussian."""
    dev = "cuda"
    L, M, nmax = c["L"], c["M"], c["nmax"]
    kT = 0.6 * (1.5 / 0.6) ** (np.arange(L) / max(1, L - 1))
    mu = -6.0 + 4.0 * np.arange(M) / max(1, M - 1)
    kT, mu = np.repeat(kT, M), np.tile(mu, L)
    N = torch.arange(nmax + 1, device=dev, dtype=torch.float64)
    mean, var = -2.0 * N - 1.5 * N * N / nmax, 0.8 * N + 1e-9
    k = torch.arange(-int(7.5 * nmax / c["e_bin"]), 1, device=dev, dtype=torch.float64)
    E = c["e_bin"] * k
    lng = (N * math.log(800.0) - torch.lgamma(N + 1))[:, None] - 0.5 * (E[None] - mean[:, None]) ** 2 / var[:, None] \
        - 0.5 * torch.log(2 * math.pi * var)[:, None]
    lng[0] = torch.where(k == 0, 0.0, -math.inf)
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    law = []
    for s in range(L * M):
        b = 1.0 / kT[s]
        x = lng - b * E[None] - (3.0 * (-0.5 * math.log(kT[s])) - b * mu[s]) * N[:, None]
        law.append(torch.softmax(x.reshape(-1), 0))
    law = torch.stack(law)
    # the bins that a run of this length reaches; each holds at least one observation
    at = torch.nonzero(law.sum(0) * c["obs"] > 2.0).reshape(-1)
    law = law[:, at]
    H = torch.zeros(L * M, len(at), device=dev, dtype=torch.float64)
    for s in range(L * M):
        H[s] = torch.bincount(torch.multinomial(law[s], c["obs"], replacement=True, generator=gen),
                              minlength=len(at)).double()
    none = torch.nonzero(H.sum(0) == 0).reshape(-1)
    H[law[:, none].argmax(0), none] = 1.0
    omega, H = H.sum(1), H.sum(0)
    q = c["Q"]
    kq, mq = np.meshgrid(np.linspace(0.65, 1.4, q), np.linspace(-5.5, -2.5, q), indexing="ij")
    return dict(kT=kT, mu=mu, omega=omega.cpu().numpy(), N=(at // E.numel()).cpu().numpy().astype(np.int32),
                E=E[at % E.numel()].cpu().numpy(), H=H.cpu().numpy(), kq=kq.ravel(), mq=mq.ravel())


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = dict(case=case)
    if kind == "mbar":
        s.update(_bins(c, seed))
        return s
    if kind == "batch":
        # the systems belong to the case, their walkers and random streams to the seed
        ps = W.uneven_batch(n_systems=c["systems"], L=c["L"], M=c["M"], seed=c["systems"], nmax_exp=(c["lo"], c["hi"]))
        gs = []
        for i, p in enumerate(ps):
            g = Regc(p.replace(seed=(seed + 7919 * i) % 65521))
            g.set_walkers(*W.uneven_initial(p, seed=seed + i))
            gs.append(g)
        b = Batch(gs, sweeps_per_step=c["sweeps"])
        b.run(5)
        b.sync()
        s.update(members=gs, batch=b, out=[_out(g) for g in gs])
        return s
    if kind == "walkers":
        g = _grid(c, seed)
        pos, n, _, sow = g.get_walkers()
        s.update(pos=_pinned(pos.shape, torch.float32), n=_pinned(n.shape, torch.int32),
                 sow=_pinned(sow.shape, torch.int32))
        s["pos"][:], s["n"][:], s["sow"][:] = pos, n, sow
        s.update(g=g, out=_out(g))
        return s
    if kind == "cycle":
        g = _grid(c, seed, 0)
        g.cycle(300, 0.99, 10)
        z = g.p.z_lo
        g.structure_init(400, 0.12, [(z, z + 0.6), (z + 0.6, z + 1.6), (z + 1.6, z + 2.6)], 49, 0.1, g.S * c["blocks"])
        s.update(g=g, out=_out(g))
        return s
    g = _grid(c, seed)
    if kind == "reweight":
        g.reset_histograms()
        g.run(c["sweeps"], 10)
        kq, mq = np.meshgrid(np.linspace(0.65, 1.4, c["Q"]), np.linspace(-5.5, -2.5, c["Q"]), indexing="ij")
        s.update(kq=kq.ravel(), mq=mq.ravel())
    if kind == "train":
        _learn(g, c["harvests"], 0, seed)
        s["seed"] = seed % 65521
    if c.get("delayed"):
        _learn(g, max(1, 16384 // (16 * g.S)), 300, seed)
        g.set_mode(True)
        g.run(20, 10)
    s.update(g=g, out=_out(g))
    return s


# ----------------------------------------------------------------- one pass

def _state(g, out):
    pos, n, e, sow = g.get_walkers(out=out)
    moves, exchanges, _ = g.counters()
    return dict(pos=pos, n=n, energy=e, state=sow, moves=moves, exchanges=exchanges)


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "sweep":
        s["g"].run(c["sweeps"] * c["blocks"], c["sweeps"])
        return _state(s["g"], s["out"])
    if kind == "cycle":
        g = s["g"]
        g.structure_reset()
        for _ in range(c["blocks"]):
            g.cycle(c["steps"], 0.99, 10)
            g.structure_sample()
        return dict(samples=g.structure_get(), **_state(g, s["out"]))
    if kind == "batch":
        s["batch"].run(c["blocks"])
        s["batch"].sync()
        got = [g.get_walkers(out=o) for g, o in zip(s["members"], s["out"])]
        return dict(pos=np.concatenate([x[0].reshape(-1) for x in got]), n=np.concatenate([x[1] for x in got]),
                    energy=np.concatenate([x[2] for x in got]), state=np.concatenate([x[3] for x in got]))
    if kind == "md":
        s["g"].cycle_md(c["steps"], 0.9, c["md_steps"], 0.005, 0.1)
        kinetic = s["g"].md(c["md_steps"], 0.005, 0.1)
        return dict(kinetic=kinetic, **_state(s["g"], s["out"]))
    if kind == "walkers":
        g = s["g"]
        g.set_walkers(s["pos"], s["n"], s["sow"])
        g.sweep(c["sweeps"])
        g.exchange()
        return list(g.get_walkers(out=s["out"]))
    if kind == "mbar":
        f, D, _ = mbar_solve(s["kT"], s["mu"], 1.0, s["omega"], s["N"], s["E"], s["H"])
        mean, pN, fq = mbar_query(s["kq"], s["mq"], 1.0, s["N"], s["E"], s["H"], D, c["nmax"])
        return dict(f=f, D=D, mean=mean, pN=pN, fq=fq)
    if kind == "reweight":
        mean, pN, f, _ = s["g"].reweight(s["kq"], s["mq"])
        return dict(mean=mean, pN=pN, f=f)
    g = s["g"]
    g.surrogate_init(s["seed"])
    for _ in range(c["harvests"]):
        g.sweep(10)
        g.surrogate_harvest(8, 8, 8.0, 0)
    loss = g.surrogate_train(c["steps"], c["batch"], 1e-3)
    X, y = g.surrogate_dataset()
    return dict(loss=loss, theta=g.surrogate_get(), X=X, y=y)


# --------------------------------------------------- what a pass cannot do without

# (mean particles as a share of nmax, pairs within the cutoff per trial move) of
# the equilibrated systems, to state a pass's bytes and operations
_TYPICAL = dict(fcc100=(0.5, 20.0), fcc111=(0.53, 14.0), two_gas=(0.5, 12.0), cluster=(0.5, 4.0), a18=(0.3, 16.0))


def work(case):
    c, kind = case, case["kind"]
    S = c["L"] * c["M"] * c.get("K", 1)
    pair = 20.0                                    # flops of one pair within the cutoff
    fill, pairs = _TYPICAL["a18" if kind == "cycle" else c.get("system", "fcc111")]
    state = S * c.get("nmax", 0) * fill * 16.0     # the configurations once
    if kind == "sweep":
        moves = S * c["sweeps"] * c["blocks"] * 20.0
        net = 2.0 * (2 * 16 * 64 + 2 * 64 * 64 + 2 * 64) + pairs * 40.0 if c.get("delayed") else 0.0
        return dict(bytes=3.0 * state + S * c["sweeps"] * c["blocks"] * 24.0, flops=moves * (pairs * pair + net))
    if kind == "cycle":
        return dict(bytes=3.0 * state + S * c["blocks"] * 1500.0,
                    flops=S * c["steps"] * c["blocks"] * 11.0 * pairs * pair)
    if kind == "batch":
        nmax = (2.0 ** (c["hi"] + 1) - 2.0 ** c["lo"]) / (c["hi"] - c["lo"] + 1)
        S *= c["systems"]
        return dict(bytes=3.0 * S * nmax * 0.3 * 16.0, flops=S * c["sweeps"] * c["blocks"] * 20.0 * pairs * pair)
    if kind == "md":
        return dict(bytes=3.0 * state * (c["steps"] + 1),
                    flops=state / 16.0 * (c["steps"] + 1) * c["md_steps"] * pairs * 2.0 * pair)
    if kind == "walkers":
        return dict(bytes=2.0 * state / 16.0 * 12.0 + 2.0 * state, flops=S * c["sweeps"] * 20.0 * pairs * pair)
    if kind == "mbar":
        B = 3.0 * c["nmax"] ** 1.5 / c["e_bin"]
        return dict(bytes=B * 28.0 + S * 24.0, flops=(S + c["Q"] ** 2) * B * 40.0)
    if kind == "reweight":
        return dict(bytes=(c["nmax"] + 1) * c["nmax"] * 30.0 * 8.0, flops=(S * 0.1 + c["Q"] ** 2) * c["nmax"] * 300.0 * 40.0)
    rows = 16.0 * S * c["harvests"]
    net = 6.0 * (16 * 64 + 64 * 64 + 64)
    return dict(bytes=rows * 68.0 * 2.0, flops=c["steps"] * c["batch"] * net + rows * 60.0 * pair)


# ------------------------------------------------------------------ in 64 bits

def exact(case, seed):
    """The reweighting in plain 64-bit torch.  The samplers' outputs are one path of a
    random process, fixed bit by bit by its seed, and training's are too: no value in
    64 bits belongs to them."""
    if case["kind"] != "mbar":
        return None
    s = _bins(case, seed)
    t = {k: torch.as_tensor(v, device="cuda", dtype=torch.float64) for k, v in s.items()}

    def u(kT, mu):
        return t["E"][None] / kT[:, None] + (-1.5 * torch.log(kT) - mu / kT)[:, None] * t["N"][None]

    us, lnom, lnH = u(t["kT"], t["mu"]), torch.log(t["omega"]), torch.log(t["H"])
    f = torch.zeros_like(lnom)

    def gradient(f):
        x = (lnom + f)[:, None] - us
        D = torch.logsumexp(x, 0)
        p = torch.exp(x - D[None])                 # a bin's share in every state
        return D, p, (p * t["H"][None]).sum(1) - t["omega"]

    def value(f):                                  # convex; its gradient is the one above
        return float((t["H"] * torch.logsumexp((lnom + f)[:, None] - us, 0)).sum() - (t["omega"] * f).sum())

    for _ in range(50):                            # the self-consistent map gets near
        D = torch.logsumexp((lnom + f)[:, None] - us, 0)
        f = -torch.logsumexp(lnH[None] - us - D[None], 1)
        f = f - f[0].clone()
    damp, last = 1e-3, value(f)
    for _ in range(300):                           # damped Newton steps to the end
        D, p, g = gradient(f)
        w = p * t["H"][None]
        hess = torch.diag(w.sum(1)) - w @ p.T
        step = torch.zeros_like(f)
        step[1:] = torch.linalg.solve(hess[1:, 1:] + damp * torch.diag(torch.diag(hess)[1:]), -g[1:])
        size = float(step.abs().max())
        new = value(f + step)
        if new <= last + 1e-12 * abs(last) or size < 1e-6:
            f, last, damp = f + step, new, (0.0 if size < 1e-3 else damp * 0.2)
            if size < 1e-13:
                break
        else:
            damp = max(damp, 1e-9) * 10.0
    D = torch.logsumexp((lnom + f)[:, None] - us, 0)
    x = lnH[None] - u(t["kq"], t["mq"]) - D[None]
    fq = -torch.logsumexp(x, 1)
    w = torch.exp(x + fq[:, None])
    pN = torch.zeros(len(fq), case["nmax"] + 1, device="cuda", dtype=torch.float64)
    pN.index_add_(1, t["N"].long(), w)
    return dict(f=f.cpu().numpy(), D=D.cpu().numpy(), mean=(w @ t["N"]).cpu().numpy(), pN=pN.cpu().numpy(),
                fq=fq.cpu().numpy())
