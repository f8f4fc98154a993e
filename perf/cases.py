"""Performance cases of the PTCA library: whole sweeps of the lattices that a
user of it runs, the batched eigenvalue call and the full-system spectrum, each
through the public entry points.

A sweep case is one Monte Carlo sweep of a chain that is under way: the state
keeps its context (schedule, workspaces, launch configuration), a pass runs
``ptca_sweep`` and reads back the spins and the record of every visit.

A PTCA_MIXED context reduces in FP32, so its free energies and eigenvalues
carry FP32 accuracy; the program stores them as float32, in the type that
holds them.  Spins, ln u and everything of an FP64 context stay float64, and
decisions are bytes.
"""
import math

import numpy as np
import torch

import paper_1502_07028_gb300 as P

DE, HUB, HOL = P.MODEL_DOUBLE_EXCHANGE, P.MODEL_HUBBARD_MF, P.MODEL_HOLSTEIN
TILED, BLOCK = P.SCHEDULE_TILED, P.SCHEDULE_BLOCK


def _sweep(name=None, **kw):
    c = dict(kind="sweep", model=DE, Lx=8, Ly=8, Lz=1, periodic=1, L_c=4, schedule=TILED, stride=0, offset=-1,
             t=1.0, coupling=8.0, mu=-6.5, T=0.05, cone=0, m_step=0.5, mixed=1, tuned=1, screen=0, observe=0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest calls: the exactly solvable toy lattice of every first
        # run, with the launch configuration a context starts with.  16 stages
        # of 4 visits: latency and launches.
        _sweep("small_8x8", tuned=0),
        # One replica of a temperature scan on 32x32, low T, sphere moves, 64
        # stages of 16 visits, default configuration, observables measured
        # after the sweep.
        _sweep("replica_32x32", Lx=32, Ly=32, L_c=8, T=0.02, tuned=0, observe=1),
        # The production lattice: 100x100, 8x8 clusters, the paper's block
        # schedule, cone moves, in the configuration the autotuner picks.
        _sweep("torus_100x100", Lx=100, Ly=100, L_c=8, schedule=BLOCK, cone=1),
        # The same lattice with the learned screen in front of the exact solves.
        _sweep("screened_100x100", Lx=100, Ly=100, L_c=8, schedule=BLOCK, cone=1, screen=1),
        # An open lattice: windows clipped at the edges, 50 <= n <= 200, ragged
        # batches, 100 stages.
        _sweep("open_100x100", Lx=100, Ly=100, periodic=0, L_c=10, stride=10, coupling=6.0, mu=-4.5, T=0.1, tuned=0),
        # The paper's own model on its largest square lattice: many small
        # matrices (n = 32).
        _sweep("hubbard_256x256", model=HUB, Lx=256, Ly=256, L_c=4, schedule=BLOCK, mu=4.0, T=0.1),
        # ... and on its largest cube, 4^3 clusters (n = 128).
        _sweep("hubbard_40x40x40", model=HUB, Lx=40, Ly=40, Lz=40, L_c=4, schedule=BLOCK, mu=4.0, T=0.15),
        # Large clusters, where the finite-cluster error has to be small: 12x12
        # (n = 288), default configuration of large contexts.
        _sweep("clusters_12x12", Lx=48, Ly=48, L_c=12, schedule=BLOCK, cone=1, tuned=0),
        # The adiabatic Holstein chain: many tiny matrices (n = 16), the
        # central update site.
        _sweep("holstein_65536", model=HOL, Lx=65536, Ly=1, L_c=8, stride=8, offset=4, coupling=1.5, mu=0.0, T=0.1),
        # The plain FP64 path, which checks and short reference chains run.
        _sweep("fp64_32x32", Lx=32, Ly=32, L_c=8, schedule=BLOCK, cone=1, mixed=0, tuned=0, observe=1),
        # The batched call: cluster matrices of 500 sites, all their
        # eigenvalues and free energies.
        dict(name="eigvals_500", kind="eigvals", Lx=32, Ly=32, L_c=8, m=500, coupling=8.0, mu=-6.5, T=0.05, mixed=1),
        # The whole lattice's one-body spectrum for a saved configuration.
        dict(name="spectrum_32x32", kind="spectrum", Lx=32, Ly=32, coupling=8.0, mixed=1),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    k = rng.choice(["torus", "torus", "open", "hubbard", "cube", "large", "chain", "fp64", "eigvals", "spectrum"])
    T = round(math.exp(rng.uniform(math.log(0.02), math.log(0.2))), 4)
    if k == "torus":
        # a two-dimensional torus of either schedule, clusters up to 8x8
        L_c = rng.randint(3, 8)
        if rng.random() < 0.5:
            Lx, Ly = (max(2 * L_c, _log(rng, 16, 110)) for _ in range(2))
            return _sweep(Lx=Lx, Ly=Ly, L_c=L_c, schedule=BLOCK, cone=rng.randint(0, 1), T=T)
        return _sweep(Lx=L_c * _log(rng, 2, 8), Ly=L_c * _log(rng, 2, 8), L_c=L_c, stride=L_c, T=T, tuned=0, observe=1)
    if k == "open":
        L_c = rng.randint(5, 10)
        return _sweep(Lx=_log(rng, 21, 100), Ly=_log(rng, 21, 100), periodic=0, L_c=L_c, stride=L_c, coupling=6.0, mu=-4.5,
                      T=T, tuned=0)
    if k == "hubbard":
        L_c = rng.randint(2, 6)
        return _sweep(model=HUB, Lx=_log(rng, 16, 200), Ly=_log(rng, 16, 200), L_c=L_c, schedule=BLOCK, mu=4.0,
                      T=max(T, 0.05))
    if k == "cube":
        L_c = rng.randint(2, 4)
        L = _log(rng, 8, 36)
        return _sweep(model=rng.choice([DE, HUB]), Lx=L, Ly=L + rng.randint(0, 3), Lz=L, L_c=L_c, schedule=BLOCK, mu=4.0,
                      T=max(T, 0.1))
    if k == "large":
        L_c = rng.randint(11, 14)
        return _sweep(Lx=2 * L_c + rng.randint(0, 9), Ly=2 * L_c + rng.randint(0, 9), L_c=L_c, schedule=BLOCK, cone=1, T=T,
                      tuned=0)
    if k == "chain":
        L_c = rng.randint(4, 16)
        return _sweep(model=rng.choice([HOL, DE]), Lx=L_c * _log(rng, 16, 4096), Ly=1, L_c=L_c, stride=L_c, offset=L_c // 2,
                      coupling=1.5, mu=0.0, T=max(T, 0.05))
    if k == "fp64":
        L_c = rng.randint(3, 8)
        return _sweep(Lx=max(2 * L_c, _log(rng, 12, 40)), Ly=max(2 * L_c, _log(rng, 12, 40)), L_c=L_c, schedule=BLOCK, T=T,
                      mixed=0, tuned=0)
    if k == "eigvals":
        L_c = rng.randint(3, 12)
        return dict(kind="eigvals", Lx=3 * L_c, Ly=2 * L_c, L_c=L_c, m=_log(rng, 20, 1500 if L_c < 9 else 300), coupling=8.0,
                    mu=-6.5, T=T, mixed=rng.randint(0, 1) if L_c < 9 else 1)
    return dict(kind="spectrum", Lx=_log(rng, 10, 36), Ly=_log(rng, 10, 36), coupling=8.0, mixed=rng.randint(0, 1))


# ---------------------------------------------------------------------------
def _config(c, seed):
    if c["kind"] == "eigvals":
        return P.Config(Lx=c["Lx"], Ly=c["Ly"], L_c=c["L_c"], stride=c["L_c"], J_H=c["coupling"], mu=c["mu"], T=c["T"],
                        precision=P.MIXED if c["mixed"] else P.FP64, seed=seed)
    if c["kind"] == "spectrum":
        return P.Config(Lx=c["Lx"], Ly=c["Ly"], L_c=4, schedule=BLOCK, J_H=c["coupling"],
                        precision=P.MIXED if c["mixed"] else P.FP64, seed=seed)
    return P.Config(Lx=c["Lx"], Ly=c["Ly"], Lz=c["Lz"], periodic=c["periodic"], L_c=c["L_c"], schedule=c["schedule"],
                    stride=c["stride"], update_offset=c["offset"], t=c["t"], J_H=c["coupling"], U=c["coupling"],
                    lam=c["coupling"], K=1.0, mu=c["mu"], T=c["T"], model=c["model"], m_step=c["m_step"],
                    proposal=P.PROPOSAL_CONE if c["cone"] else P.PROPOSAL_SPHERE, cone_deg=30.0,
                    precision=P.MIXED if c["mixed"] else P.FP64, seed=seed)


def _start(c, seed):
    """The configuration a chain starts from: unit spins, mean fields of
    length 0.6 to 1.1, or distortions in [-1, 1]."""
    g = np.random.default_rng([seed, 15])
    N = c["Lx"] * c["Ly"] * c.get("Lz", 1)
    if c.get("model", DE) == HOL:
        S = np.zeros((N, 3))
        S[:, 0] = g.uniform(-1.0, 1.0, N)
        return S
    S = g.normal(size=(N, 3))
    S /= np.linalg.norm(S, axis=1, keepdims=True)
    return S * g.uniform(0.6, 1.1, (N, 1)) if c.get("model", DE) == HUB else S


def _weights(seed):
    """Surrogate weights as a program that saved a trained network loads them."""
    g = np.random.default_rng([seed, 16])
    parts = []
    for rows, cols in ((256, 160), (256, 256), (256, 256), (8, 256)):
        parts += [(g.normal(size=(rows, cols)) / math.sqrt(cols)).ravel(), np.zeros(rows)]
    return torch.from_numpy(np.concatenate(parts).astype(np.float32)).cuda()


def prepare(case, seed):
    cfg = _config(case, seed)
    ctx = P.Context(cfg)
    S = _start(case, seed)
    ctx.set_spins(torch.from_numpy(S))
    st = {"ctx": ctx, "case": case}
    if case["kind"] == "spectrum":
        st["eig"] = torch.empty(2 * cfg.N, dtype=torch.float64, device="cuda")
        return st
    if case["kind"] == "eigvals":
        st["sites"] = torch.from_numpy((np.arange(case["m"]) * 7 % cfg.N).astype(np.int32)).cuda()
        return st
    if case["tuned"]:
        # what the autotuner settles on for these orders
        n = 2 * case["L_c"] ** ((case["Lx"] > 1) + (case["Ly"] > 1) + (case["Lz"] > 1))
        if n <= 128:
            P.ptca_set_launch_config(ctx.h, P.PIPELINE_OVERLAP if case["schedule"] == BLOCK else P.PIPELINE_STAGES,
                                     1 if n <= 32 else 4)
    if case["screen"]:
        theta = _weights(seed)
        P.ptca_surrogate_init(ctx.h, 1)
        P.ptca_surrogate_set_params(ctx.h, theta, 0.05)
        P.ptca_surrogate_enable(ctx.h, True)
    N = cfg.N
    new = lambda dt, *sh: torch.empty(sh or (N,), dtype=dt, device="cuda")  # noqa: E731
    st.update(site=new(torch.int32), lnu=new(torch.float64), acc=new(torch.uint8), Fo=new(torch.float64),
              Fn=new(torch.float64), S=new(torch.float64, N, 3))
    return st


def run(st):
    ctx, case = st["ctx"], st["case"]
    f = (lambda x: x.float()) if case["mixed"] else (lambda x: x)
    if case["kind"] == "spectrum":
        # the double-float reduction of a mixed context is FP64-class
        P.ptca_full_spectrum(ctx.h, st["eig"])
        return {"eig": st["eig"]}
    if case["kind"] == "eigvals":
        H, off, n = ctx.build_clusters(st["sites"])
        eig, eoff = ctx.cluster_eigvals(H, off, n)
        F = ctx.free_energy(eig, eoff, n)
        return {"eig": f(eig), "F": f(F), "n": n}
    P.ptca_sweep(ctx.h, 1, stats=False)
    P.ptca_get_spins(ctx.h, st["S"])
    P.ptca_sweep_record(ctx.h, st["site"], st["Fo"], st["Fn"], st["lnu"], st["acc"])
    out = {"spins": st["S"], "site": st["site"], "lnu": st["lnu"], "accepted": st["acc"], "F_old": f(st["Fo"]),
           "F_new": f(st["Fn"])}
    if case["observe"]:
        o = ctx.observables()
        out["S_q"] = np.array([o.S_00, o.S_pipi])
        out["F_site"], out["filling"], out["acceptance"] = (
            np.array([x], np.float32 if case["mixed"] else np.float64) for x in (o.F_site, o.filling, o.acceptance))
    return out


def work(case):
    """Bytes: spins in and out and the records of a sweep (its matrices are
    built on the fly); matrices and eigenvalues of a batch.  Operations: the
    (16/3) n^3 of a values-only Hermitian reduction, once for each visit (its
    two matrices differ in one site's block)."""
    if case["kind"] == "spectrum":
        n = 2 * case["Lx"] * case["Ly"]
        return {"bytes": 24 * n // 2 + 8 * n, "flops": 16 / 3 * n ** 3}
    if case["kind"] == "eigvals":
        n, m = 2 * case["L_c"] ** 2, case["m"]
        return {"bytes": m * (n * (n + 1) / 2 * (8 if case["mixed"] else 16) + 8 * n + 8), "flops": m * 16 / 3 * n ** 3}
    N = case["Lx"] * case["Ly"] * case["Lz"]
    flops = 0.0
    if case["periodic"]:
        n = 2 * case["L_c"] ** ((case["Lx"] > 1) + (case["Ly"] > 1) + (case["Lz"] > 1))
        flops = N * 16 / 3 * n ** 3
    else:
        o, L_c = case["L_c"] // 2, case["L_c"]
        ext = [np.array([min(c - o + L_c - 1, L - 1) - max(c - o, 0) + 1 for c in range(L)], float)
               for L in (case["Lx"], case["Ly"])]
        flops = 16 / 3 * 8 * (ext[0] ** 3).sum() * (ext[1] ** 3).sum()
    return {"bytes": N * (48 + 29), "flops": flops}


# ---------------------------------------------------------------------------
# The same results in plain numpy, 64 bits.
def _philox(seed, sweep, site, purpose):
    M = 0xFFFFFFFF
    u = np.uint64
    x = [site.astype(u), np.full_like(site, purpose, dtype=u), np.full_like(site, sweep & M, dtype=u),
         np.full_like(site, sweep >> 32, dtype=u)]
    k0, k1 = seed & M, (seed >> 32) & M
    for _ in range(10):
        p0, p1 = u(0xD2511F53) * x[0], u(0xCD9E8D57) * x[2]
        x = [(p1 >> u(32)) ^ x[1] ^ u(k0), p1 & u(M), (p0 >> u(32)) ^ x[3] ^ u(k1), p0 & u(M)]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    a, b = x[0] | (x[1] << u(32)), x[2] | (x[3] << u(32))
    return tuple(((h >> u(11)).astype(np.float64) + 0.5) * 2.0 ** -53 for h in (a, b))


def _propose(c, seed, sites, S):
    u0, u1 = _philox(seed, 0, sites, 1)
    old = S[sites]
    if c["model"] == HOL:
        new = old.copy()
        new[:, 0] += c["m_step"] * (2 * u0 - 1)
        return new
    z, az = 2 * u0 - 1, 2 * np.pi * u1
    r = np.sqrt(np.maximum(0, 1 - z * z))
    d = np.stack([r * np.cos(az), r * np.sin(az), z], 1)
    if c["model"] == HUB:
        return old + c["m_step"] * np.cbrt(_philox(seed, 0, sites, 4)[0])[:, None] * d
    if not c["cone"]:
        return d
    ct = 1 - u0 * (1 - math.cos(math.radians(30.0)))
    st = np.sqrt(np.maximum(0, 1 - ct * ct))
    v = np.stack([st * np.cos(az), st * np.sin(az), ct], 1)
    a, b, cc = old.T
    k = 1 / (1 + cc)
    out = np.stack([(1 - a * a * k) * v[:, 0] - a * b * k * v[:, 1] + a * v[:, 2],
                    -a * b * k * v[:, 0] + (1 - b * b * k) * v[:, 1] + b * v[:, 2],
                    -a * v[:, 0] - b * v[:, 1] + cc * v[:, 2]], 1)
    low = cc < -1 + 1e-12
    out[low] = v[low] * [1, -1, -1]
    return out / np.linalg.norm(out, axis=1, keepdims=True)


def _stages(c):
    L = (c["Lx"], c["Ly"], c["Lz"])
    if c["schedule"] == BLOCK:
        cuts = [[range(n)] if n == 1 else [range((n + 1) // 2), range((n + 1) // 2, n)] for n in L]
    else:
        s = c["stride"] or c["L_c"]
        cuts = [[range(n)] if n == 1 else [range(a, n, s) for a in range(min(s, n))] for n in L]
    for zs in cuts[2]:
        for ys in cuts[1]:
            for xs in cuts[0]:
                got = np.array([(z * L[1] + y) * L[0] + x for z in zs for y in ys for x in xs], dtype=np.int64)
                if got.size:
                    yield got


def _windows(c, sites):
    """Groups of visits whose windows have one shape: (visits, extents, lattice
    sites of each window)."""
    L, L_c = (c["Lx"], c["Ly"], c["Lz"]), c["L_c"]
    o = c["offset"] if c["offset"] >= 0 else (L_c // 2 if c["schedule"] == TILED else 0)
    pos = (sites % L[0], sites // L[0] % L[1], sites // (L[0] * L[1]))
    start, ext = [], []
    for n, p in zip(L, pos):
        lo, hi = (np.zeros_like(p), np.zeros_like(p)) if n == 1 else (p - o, p - o + L_c - 1)
        if not c["periodic"]:
            lo, hi = np.maximum(lo, 0), np.minimum(hi, n - 1)
        start.append(lo)
        ext.append(hi - lo + 1)
    key = (ext[2] * 1000 + ext[1]) * 1000 + ext[0]
    for q in np.unique(key):
        at = np.nonzero(key == q)[0]
        e = [int(x[at[0]]) for x in ext]
        axes = [(start[a][at][:, None] + np.arange(e[a])) % L[a] for a in range(3)]
        g = (axes[2][:, :, None, None] * L[1] + axes[1][:, None, :, None]) * L[0] + axes[0][:, None, None, :]
        yield at, e, g.reshape(len(at), -1)


def _hamiltonian(c, e, v, periodic):
    m, ns = v.shape[:2]
    J = {DE: c["coupling"], HUB: c["coupling"] / 2, HOL: 0.0}[c.get("model", DE)]
    d = {DE: 0 * v[..., 0], HUB: 0 * v[..., 0] + c["coupling"] / 2, HOL: c["coupling"] * v[..., 0]}[c.get("model", DE)]
    H = np.zeros((m, ns, 2, ns, 2), dtype=np.complex128)
    i = np.arange(ns)
    H[:, i, 0, i, 0] = d - J * v[..., 2]
    H[:, i, 1, i, 1] = d + J * v[..., 2]
    H[:, i, 1, i, 0] = -J * (v[..., 0] + 1j * v[..., 1])
    H[:, i, 0, i, 1] = -J * (v[..., 0] - 1j * v[..., 1])
    idx = i.reshape(e[2], e[1], e[0])
    for ax, n in ((2, e[0]), (1, e[1]), (0, e[2])):
        a, b = idx, np.roll(idx, -1, axis=ax)
        if not (periodic and n >= 2):
            a, b = np.delete(a, -1, axis=ax), np.delete(b, -1, axis=ax)
        for p, q in zip(a.ravel(), b.ravel()):
            for s in (0, 1):
                H[:, p, s, q, s] -= c.get("t", 1.0)
                H[:, q, s, p, s] -= c.get("t", 1.0)
    return H.reshape(m, 2 * ns, 2 * ns)


def _eigvalsh(H, chunk=64):
    return np.concatenate([np.linalg.eigvalsh(H[k:k + chunk]) for k in range(0, len(H), chunk)])


def _free(e, mu, T):
    x = -(e - mu) / T
    return -T * (np.maximum(x, 0) + np.log1p(np.exp(-np.abs(x)))).sum(-1)


def _classical(c, v):
    m2 = (v ** 2).sum(-1)
    if c["model"] == HUB:
        return (c["coupling"] / 4 * (m2 - 1)).sum(-1)
    if c["model"] == HOL:
        return (0.5 * m2 - c["coupling"] * v[..., 0] + c["mu"]).sum(-1)
    return 0.0


def exact(case, seed):
    if case["kind"] == "spectrum":
        if case["Lx"] * case["Ly"] > 1100:
            return None
        v = _start(case, seed)[None]
        return {"eig": np.linalg.eigvalsh(_hamiltonian(case, [case["Lx"], case["Ly"], 1], v, True)[0])}
    S = _start(case, seed)
    if case["kind"] == "eigvals":
        if case["m"] * (2 * case["L_c"] ** 2) ** 3 > 2.5e9:
            return None
        c = dict(case, Lz=1, periodic=1, offset=-1, schedule=TILED)
        sites = np.arange(case["m"]) * 7 % (case["Lx"] * case["Ly"])
        eig, F = np.empty((case["m"], 2 * case["L_c"] ** 2)), np.empty(case["m"])
        for at, e, g in _windows(c, sites):
            eig[at] = _eigvalsh(_hamiltonian(c, e, S[g], True))
        return {"eig": eig, "F": _free(eig, case["mu"], case["T"]), "n": None}
    if case["screen"] or work(case)["flops"] > 16 / 3 * 2.2e9:
        return None
    site, lnu, acc, Fo, Fn, per, fill = [], [], [], [], [], [], []
    for sites in _stages(case):
        new = _propose(case, seed, sites, S)
        u = np.log(_philox(seed, 0, sites, 2)[0])
        F, fl, n_c = np.empty((2, sites.size)), np.empty((2, sites.size)), np.empty(sites.size)
        for at, e, g in _windows(case, sites):
            v = S[g]
            for k in range(2):
                if k:
                    v = np.where((g == sites[at][:, None])[..., None], new[at][:, None], v)
                eig = _eigvalsh(_hamiltonian(case, e, v, bool(case["periodic"])))
                F[k, at] = _free(eig, case["mu"], case["T"]) + _classical(case, v)
                fl[k, at] = (0.5 - 0.5 * np.tanh(0.5 * (eig - case["mu"]) / case["T"])).sum(-1)
                n_c[at] = g.shape[1]
        ok = u < -(F[1] - F[0]) / case["T"]
        S = S.copy()
        S[sites[ok]] = new[ok]
        site.append(sites), lnu.append(u), acc.append(ok), Fo.append(F[0]), Fn.append(F[1])
        per.append(np.where(ok, F[1], F[0]) / n_c), fill.append(np.where(ok, fl[1], fl[0]) / n_c)
    cat = np.concatenate
    out = {"spins": S, "site": None, "lnu": cat(lnu), "accepted": None, "F_old": cat(Fo), "F_new": cat(Fn)}
    if case["observe"]:
        i = np.arange(len(S))
        sign = 1.0 - 2.0 * ((i % case["Lx"] + i // case["Lx"] % case["Ly"] + i // (case["Lx"] * case["Ly"])) % 2)
        out["S_q"] = np.array([(S.mean(0) ** 2).sum(), ((S * sign[:, None]).mean(0) ** 2).sum()])
        out["F_site"], out["filling"], out["acceptance"] = (np.array([cat(x).mean()]) for x in (per, fill, acc))
    return out
