"""The measured workloads of the library: what a simulation program has it do, through the public
entry points of the Python binding.

Kinds of case
  kspace   one k-space evaluation of a snapshot (`Context.forces_virial`, `forces_virial_xyzq`, or
           the host-buffer call), FP64 or FP32-phase, on the seeded systems of `inputs.py`
  batched  one evaluation of many uneven systems (`Batch.evaluate`)
  npt      a short isotropic Langevin NPT run of one replica from a stored configuration
           (`NptReplica.init`, `.step`)
  water    the same for rigid 3-site water (`WaterReplica`)
  serve    a handful of replica requests through the serving loop (`Server`), submission to results
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2110_14362_gb300 as rbe
from paper_2110_14362_gb300 import inputs

KB = 0.00831446261815324   # kJ/mol/K
BAR = 6.02214076e-5        # kJ/mol/A^3
KE = 1389.35457644382      # kJ/mol A/e^2
WATER_MASS = (15.9994, 1.008, 1.008)


# ---------------------------------------------------------------------------------
# The cases.

def listed():
    return [
        # the small snapshot of the accuracy checks, on the reference-accuracy path: an evaluation
        # whose cost is launches and latency
        dict(name="snapshot_fp64", kind="kspace", system="snapshot", precision="fp64", input="f64", N=1000, P=100),
        # the smallest replicas of a serving stream fed with float32 (x, y, z, q) records, a ragged N
        dict(name="small_xyzq_fp32", kind="kspace", system="uniform", precision="fp32", input="xyzq", N=4099, P=100),
        # the membrane-like slab on both paths: the ordinary mid-size evaluation, and the FP64 run it
        # is checked against
        dict(name="slab_fp32", kind="kspace", system="slab", precision="fp32", input="f64", N=300000, P=200),
        dict(name="slab_fp64", kind="kspace", system="slab", precision="fp64", input="f64", N=300000, P=200),
        # the middle of the large-N sweep, FP64 throughout
        dict(name="sweep_fp64", kind="kspace", system="uniform", precision="fp64", input="f64", N=1000000, P=500),
        # the largest point of the sweep, the headline workload of the benchmark
        dict(name="sweep_fp32", kind="kspace", system="uniform", precision="fp32", input="f64", N=4000000, P=2000),
        # an engine that keeps its particles in (pinned) host memory and calls the evaluation each step
        dict(name="host_fp32", kind="kspace", system="uniform", precision="fp32", input="host", N=1000000, P=500),
        # the k-space of 64 uneven replicas of 1e3 to 1e5 charges in one call
        dict(name="batched_64", kind="batched", items=64, P=100, n_hi=1e5),
        # one replica of the serving stream's mean size: ten NPT steps with a neighbour list
        dict(name="npt_fp32", kind="npt", precision="fp32", N=20000, P=100, steps=10, skin=1.0),
        # the same system one at a time on the FP64 path, the run that the served form is compared with
        dict(name="npt_fp64", kind="npt", precision="fp64", N=20000, P=100, steps=4, skin=1.0),
        # the plain-method run: 3000 rigid 3-site waters, FP64 (alpha where the batch holds 300 K)
        dict(name="water_fp64", kind="water", molecules=3000, P=100, steps=4, alpha=0.08),
        # continuous batching: twelve requests of uneven N through the serving loop
        dict(name="serve_fp32", kind="serve", requests=12, steps=20, chunk=10, slots=8, P=100, n_hi=1e5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["kspace", "kspace", "kspace", "kspace", "batched", "npt", "npt", "water", "serve"])
    if kind == "kspace":
        precision = rng.choice(["fp64", "fp32"])
        inp = "f64" if precision == "fp64" else rng.choice(["f64", "f64", "xyzq", "host"])
        P = _log_int(rng, 50, 2000)
        most = 5e8 if precision == "fp64" else (5e8 if inp == "host" else 8e9)
        N = _log_int(rng, 1000, min(4e6 if precision == "fp32" else 1e6, most / P))
        return dict(kind=kind, system=rng.choice(["uniform", "uniform", "slab"]), precision=precision, input=inp, N=N, P=P)
    if kind == "batched":
        return dict(kind=kind, items=rng.randint(5, 64), P=_log_int(rng, 60, 300), n_hi=float(_log_int(rng, 1e4, 1e5)))
    if kind == "npt":
        precision = rng.choice(["fp64", "fp32"])
        return dict(kind=kind, precision=precision, N=_log_int(rng, 3500, 1e5 if precision == "fp32" else 3e4),
                    P=_log_int(rng, 60, 300), steps=rng.randint(2, 12 if precision == "fp32" else 5),
                    skin=rng.choice([0.0, 1.0, 1.0]))
    if kind == "water":
        return dict(kind=kind, molecules=_log_int(rng, 400, 3000), P=_log_int(rng, 60, 200), steps=rng.randint(1, 4),
                    alpha=round(rng.uniform(0.07, 0.1), 4))
    return dict(kind=kind, requests=rng.randint(3, 12), steps=rng.choice([10, 15, 20]), chunk=rng.choice([5, 10]),
                slots=rng.randint(2, 8), P=_log_int(rng, 60, 200), n_hi=float(_log_int(rng, 1e4, 1e5)))


# ---------------------------------------------------------------------------------
# Inputs.

def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _gpu(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64).to(_device())


def _snapshot(case, seed):
    """Positions, charges, box and alpha of a k-space case (float32-rounded for the xyzq records)."""
    N = case["N"]
    if case["system"] == "snapshot":
        s = inputs.small_snapshot(seed)
    elif case["system"] == "slab":
        f = (N / 300000.0) ** (1.0 / 3.0)  # the slab's density and proportions at any N
        s = inputs.slab(N, seed, box=(80.0 * f, 80.0 * f, 120.0 * f), sigma_z=10.0 * f, half_width=20.0 * f, P=case["P"])
    else:
        s = inputs.uniform_density(N, 0.1, seed, P=case["P"])
    pos, q = s.pos, s.q
    if case["input"] == "xyzq":
        pos, q = pos.astype(np.float32), q.astype(np.float32)
    return pos, q, s.box, s.alpha


def _replica_sizes(n, n_hi, seed):
    rng = np.random.default_rng(seed)
    return [2 * int(math.exp(rng.uniform(math.log(1e3), math.log(n_hi))) / 2) for _ in range(n)]


def _batch_systems(case, seed):
    out = []
    # the sizes are the case's, the same for every seed (the first requests of one stream)
    for k, N in enumerate(_replica_sizes(case["items"], case["n_hi"], 11)):
        pos, _, q, _, box = inputs.npt_replica(N, seed * 1000 + k)
        out.append((pos, q, box, 1000 + 7 * seed + k))
    return out


def _npt_params(box, skin):
    return rbe.NptParams(dt=0.001, kT=KB * 300.0, P_ext=BAR, gamma=10.0, gamma_V=2.0,
                         M_V=rbe.piston_mass(0.5, 4.5e-5 / BAR, float(np.prod(box))), rc=7.0, qqr2e=KE / 78.5,
                         lj_sigma=2.0, lj_eps=0.5, max_disp=0.05, kspace=1, real=1, noise=1, barostat=1, skin=skin)


def _water_system(case, seed):
    s = inputs.water(case["molecules"], seed)
    n = case["molecules"]
    mass = np.tile(WATER_MASS, n)
    mom = np.random.default_rng(seed + 7).standard_normal((3 * n, 3)) * np.sqrt(KB * 300.0 * 100.0 * mass)[:, None]
    prm = rbe.NptParams(dt=0.001, kT=KB * 300.0, P_ext=BAR, gamma=10.0, gamma_V=2.0,
                        M_V=rbe.piston_mass(0.5, 4.5e-5 / BAR, float(np.prod(s.box))), rc=10.0, qqr2e=KE,
                        lj_sigma=3.166, lj_eps=0.650, max_disp=0.05, kspace=1, real=1, noise=1, barostat=1)
    return s.pos, mom, s.q, mass, s.box, prm


def _serve_requests(case, seed):
    out = []
    for k, N in enumerate(_replica_sizes(case["requests"], case["n_hi"], 5)):
        pos, mom, q, mass, box = inputs.npt_replica(N, seed * 1000 + k)
        out.append((pos, mom, q, mass, box, _npt_params(box, 1.0), 2000 + 13 * seed + k))
    return out


_PRECISION = {"fp64": rbe.RBE_FP64, "fp32": rbe.RBE_FP32_PHASE}


def prepare(case, seed):
    kind, dev = case["kind"], _device()
    stream = torch.cuda.current_stream().cuda_stream
    key = 12345 + seed
    if kind == "kspace":
        pos, q, box, alpha = _snapshot(case, seed)
        ctx = rbe.Context(box, alpha, case["P"], key, _PRECISION[case["precision"]], stream=stream)
        N = q.shape[0]
        if case["input"] == "host":
            pin = lambda a: torch.as_tensor(a).pin_memory()  # noqa: E731
            keep = (pin(pos), pin(q), torch.empty((N, 3), dtype=torch.float64).pin_memory())
            return dict(case=case, ctx=ctx, keep=keep, args=tuple(t.numpy() for t in keep))
        F = torch.empty((N, 3), dtype=torch.float64, device=dev)
        W = torch.empty(9, dtype=torch.float64, device=dev)
        E = torch.empty(2, dtype=torch.float64, device=dev)
        if case["input"] == "xyzq":
            args = (torch.as_tensor(np.column_stack([pos, q])).to(dev).contiguous(),)
        else:
            args = (_gpu(pos), _gpu(q))
        return dict(case=case, ctx=ctx, args=args, out=(F, W, E))
    if kind == "batched":
        made = _batch_systems(case, seed)
        # one buffer for all items' forces, virials and energies, an item's part behind the one before
        F = torch.empty((sum(len(s[1]) for s in made), 3), dtype=torch.float64, device=dev)
        W = torch.empty((len(made), 9), dtype=torch.float64, device=dev)
        E = torch.empty((len(made), 2), dtype=torch.float64, device=dev)
        systems, at = [], 0
        for k, (pos, q, box, sd) in enumerate(made):
            systems.append(dict(pos=_gpu(pos), q=_gpu(q), F=F[at:at + len(q)], W=W[k], E=E[k], box=box, seed=sd, step=0))
            at += len(q)
        b = rbe.Batch(0.2, case["P"], len(systems), 1.01 * max(float(s["box"][0]) for s in systems), stream=stream)
        return dict(case=case, batch=b, systems=systems, items=b.items(systems), out=(F, W, E))
    if kind in ("npt", "water"):
        if kind == "npt":
            pos, mom, q, mass, box = inputs.npt_replica(case["N"], seed)
            ctx = rbe.Context(box, 0.2, case["P"], key, _PRECISION[case["precision"]], stream=stream)
            rep = rbe.NptReplica(pos, mom, q, mass, box, _npt_params(box, case["skin"]), dev)
        else:
            pos, mom, q, mass, box, prm = _water_system(case, seed)
            ctx = rbe.Context(box, case["alpha"], case["P"], key, rbe.RBE_FP64, stream=stream)
            rep = rbe.WaterReplica(pos, mom, q, mass, box, prm, dev)
        start = (rep.pos.clone(), rep.mom.clone(), rep.cell.clone())
        return dict(case=case, ctx=ctx, rep=rep, start=start)
    srv = rbe.Server(0.2, case["P"], max_slots=case["slots"], chunk_steps=case["chunk"], mem_budget=64 << 30)
    return dict(case=case, server=srv, requests=_serve_requests(case, seed))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "kspace":
        ctx = state["ctx"]
        if case["input"] == "host":
            pos, q, F = state["args"]
            F, W, E = rbe.rbe_kspace_forces_virial_host(ctx.h, pos, q, 3, F)
            return {"forces": F, "virial": W.reshape(9), "energy": E}
        F, W, E = state["out"]
        if case["input"] == "xyzq":
            ctx.forces_virial_xyzq(state["args"][0], 3, F, W, E)
        else:
            ctx.forces_virial(state["args"][0], state["args"][1], 3, F, W, E)
        return {"forces": F, "virial": W, "energy": E}
    if kind == "batched":
        state["batch"].evaluate(state["items"])
        F, W, E = state["out"]
        return {"forces": F, "virial": W, "energy": E}
    if kind in ("npt", "water"):
        rep, ctx = state["rep"], state["ctx"]
        for to, of in zip((rep.pos, rep.mom, rep.cell), state["start"]):
            to.copy_(of)
        rep.sys.step = 0
        rep.init(ctx)
        rep.step(ctx, case["steps"])
        return {"pos": rep.pos, "mom": rep.mom, "force": rep.force, "cell": rep.cell}
    srv = state["server"]
    ids = [srv.submit(pos, mom, q, mass, box, prm, sd, case["steps"])
           for pos, mom, q, mass, box, prm, sd in state["requests"]]
    while True:
        queued, active, _ = srv.progress(wait=True)
        if queued == 0 and active == 0:
            break
    got = [srv.result(i) for i in ids]
    return {"pos": [g[0] for g in got], "mom": [g[1] for g in got], "cell": [g[2] for g in got]}


# ---------------------------------------------------------------------------------
# What a pass cannot do without.  Per (particle, frequency) pair: the phase m.s (5 operations), a
# sine and a cosine and their two products into rho (6), and again the phase, one sine of the
# shifted phase and three products into the force (12): 23.  Per real-space pair within the cutoff
# (each once): separation, distance, Coulomb and Lennard-Jones terms, force and virial sums: 60.

def _kspace_work(N, P, in_bytes=32):
    return N * (in_bytes + 24) + 16 * P + 88, 23.0 * N * P


def _npt_step_work(N, P, rc, density):
    b, f = _kspace_work(N, P)
    # state read and written (r, p, F, masses), the forces of both parts
    return b + N * 160, f + N * (60.0 * 0.5 * density * 4.0 / 3.0 * math.pi * rc ** 3 + 150.0)


def work(case):
    kind = case["kind"]
    if kind == "kspace":
        b, f = _kspace_work(case["N"], case["P"], 16 if case["input"] == "xyzq" else 32)
        return {"bytes": b, "flops": f}
    if kind == "batched":
        parts = [_kspace_work(N, case["P"]) for N in _replica_sizes(case["items"], case["n_hi"], 11)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if kind == "npt":
        b, f = _npt_step_work(case["N"], case["P"], 7.0, 0.1)
        return {"bytes": b * (case["steps"] + 1), "flops": f * (case["steps"] + 1)}
    if kind == "water":
        N = 3 * case["molecules"]
        b, f = _npt_step_work(N, case["P"], 10.0, 3 * 0.602214076 / 18.01528)
        return {"bytes": b * (case["steps"] + 1), "flops": f * (case["steps"] + 1)}
    parts = [_npt_step_work(N, case["P"], 7.0, 0.1) for N in _replica_sizes(case["requests"], case["n_hi"], 5)]
    return {"bytes": sum(p[0] for p in parts) * (case["steps"] + 1),
            "flops": sum(p[1] for p in parts) * (case["steps"] + 1)}


# ---------------------------------------------------------------------------------
# The same results in 64 bits, in plain numpy and torch.

_MASK = (1 << 32) - 1


def _philox(c0, c1, c2, c3, seed):
    """Philox-4x32-10 on uint64 arrays of 32-bit words."""
    c = [np.asarray(x, dtype=np.uint64) for x in np.broadcast_arrays(c0, c1, c2, c3)]
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK
    m = np.uint64(_MASK)
    for r in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m]
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return c


def _sample(box, alpha, P, seed, step):
    """The sampled frequencies (P x 3) and S: per-axis discrete Gaussians by inverse CDF on integer
    cumulative weights, redrawn while zero."""
    rows, H = [], 1.0
    for ell in box:
        c = (math.pi * math.pi) / (alpha * (float(ell) * float(ell)))
        M = math.ceil(math.sqrt(60.0 * 0.69314718055994530942 / c))
        sh = 62 - (2 * M + 1).bit_length()
        w = [int(round(math.ldexp(math.exp(-c * a * a), sh))) for a in range(M + 1)]
        cum = np.cumsum(np.array([w[abs(j - M)] for j in range(2 * M + 1)], dtype=np.uint64))
        rows.append((M, cum))
        H *= math.ldexp(float(int(cum[-1])), -sh)
    out = np.zeros((P, 3), dtype=np.int64)
    left = np.arange(P)
    attempt = 0
    while left.size:
        w0 = _philox(left, 2 * attempt, step & _MASK, (step >> 32) & 0xFFFFFF, seed)
        w1 = _philox(left, 2 * attempt + 1, step & _MASK, (step >> 32) & 0xFFFFFF, seed)
        u = [(w0[0], w0[1]), (w0[2], w0[3]), (w1[0], w1[1])]
        for t, (M, cum) in enumerate(rows):
            U = (u[t][0] << np.uint64(21)) | (u[t][1] >> np.uint64(11))
            total = int(cum[-1])
            T = np.array([(int(x) * total) >> 53 for x in U], dtype=np.uint64)
            out[left, t] = np.searchsorted(cum, T, side="right") - M
        left = left[~out[left].any(axis=1)]
        attempt += 1
    return out, H - 1.0


def _kspace(pos, q, box, alpha, m, S):
    """Forces, virial and energies of the sampled frequencies (torch, FP64, in chunks of particles)."""
    dev, P, N = pos.device, m.shape[0], pos.shape[0]
    L = torch.as_tensor(np.asarray(box, dtype=np.float64), device=dev)
    V = float(L.prod())
    mt = torch.as_tensor(m, dtype=torch.float64, device=dev)
    k = 2.0 * math.pi * mt / L
    kk = (k * k).sum(1)
    re, im = (torch.zeros(P, dtype=torch.float64, device=dev) for _ in range(2))
    chunk = max(1, int(1e8) // P)

    def angle(a):
        s = pos[a:a + chunk] / L
        t = (s - torch.floor(s)) @ mt.T
        return (t - torch.round(t)).mul_(2.0 * math.pi)

    for a in range(0, N, chunk):
        th, qa = angle(a), q[a:a + chunk]
        re += qa @ torch.cos(th)
        im += qa @ torch.sin(th)
    beta = (S / P) * 4.0 * math.pi / (V * kk)
    F = torch.empty_like(pos)
    for a in range(0, N, chunk):
        th = angle(a)
        g = torch.sin(th) * (beta * re) - torch.cos(th) * (beta * im)
        F[a:a + chunk] = q[a:a + chunk, None] * (g @ k)
    e = (2.0 * math.pi / V) * (S / P) * (re * re + im * im) / kk
    W = torch.eye(3, dtype=torch.float64, device=dev) * e.sum() - \
        2.0 * (k * (e * (1.0 / kk + 0.25 / alpha))[:, None]).T @ k
    E = torch.stack([e.sum(), -math.sqrt(alpha / math.pi) * (q * q).sum()])
    return F, W.reshape(9), E


def _normals(seed, stream, step, index):
    w = _philox(index, 0, step & _MASK, (stream << 24) | ((step >> 32) & 0xFFFFFF), seed)
    u = [(x.astype(np.float64) + 0.5) * 2.0 ** -32 for x in w]
    z = []
    for a in (0, 2):
        r = np.sqrt(-2.0 * np.log(u[a]))
        z += [r * np.cos(2.0 * math.pi * u[a + 1]), r * np.sin(2.0 * math.pi * u[a + 1])]
    return z


def _expm1_over(x, t):
    return t * (1.0 + x * (0.5 + x / 6.0)) if abs(x) < 1e-8 else t * math.expm1(x) / x


def _pairs_within(pos, L, r):
    """Index pairs i < j within r (nearest image), by brute force in chunks."""
    N, got = pos.shape[0], []
    p32 = (pos - L * torch.floor(pos / L)).float()
    chunk = max(1, int(2e8) // N)
    for a in range(0, N, chunk):
        d2 = 0.0
        for t in range(3):
            d = (p32[a:a + chunk, t, None] - p32[None, :, t]).abs_()
            d2 = torch.minimum(d, L - d).square_() + d2
        i, j = torch.nonzero(d2 < r * r, as_tuple=True)
        i = i + a
        got.append(torch.stack([i[i < j], j[i < j]]))
    return torch.cat(got, 1)


def _pair_forces(pos, q, L, alpha, prm, pairs, lj_mask):
    """erfc Coulomb and Lennard-Jones within rc: forces, virial trace, both energies."""
    i, j = pairs
    d = pos[j] - pos[i]
    d = d - L * torch.round(d / L)
    r2 = (d * d).sum(1)
    on = r2 < prm.rc ** 2
    i, j, d, r2 = i[on], j[on], d[on], r2[on]
    lj = torch.ones_like(r2) if lj_mask is None else lj_mask[on].double()
    r, sa = r2.sqrt(), math.sqrt(alpha)
    qq, ec = prm.qqr2e * q[i] * q[j], torch.erfc(sa * r)
    s6 = (prm.lj_sigma ** 2 / r2) ** 3
    f = qq * (ec / r2 + 2.0 * sa * torch.exp(-alpha * r2) / (math.sqrt(math.pi) * r)) / r + \
        lj * 24.0 * prm.lj_eps * (2.0 * s6 * s6 - s6) / r2
    F = torch.zeros_like(pos).index_add_(0, j, f[:, None] * d).index_add_(0, i, -f[:, None] * d)
    return F, float((f * r2).sum()), float((qq * ec / r).sum()), float((lj * 4.0 * prm.lj_eps * (s6 * s6 - s6)).sum())


def _cap(d, cap):
    n = d.norm(dim=1, keepdim=True)
    return torch.where(n > cap, d * (cap / n), d)


def _npt(pos, mom, q, mass, box, prm, alpha, P, seed, steps):
    """The isotropic NPT steps of one replica in FP64."""
    r, p, q, m = (_gpu(a) for a in (pos, mom, q, mass))
    m1, L, pV = m[:, None], float(box[0]), 0.0
    pairs = _pairs_within(r, L, prm.rc + 0.3 + 0.1 * steps)

    def forces(step):
        mk, S = _sample([L] * 3, alpha, P, seed, step)
        Fk, Wk, Ek = _kspace(r, q, [L] * 3, alpha, mk, S)
        Fr, Wr, Ec, El = _pair_forces(r, q, L, alpha, prm, pairs, None)
        return prm.qqr2e * Fk + Fr, prm.qqr2e * float(Wk[0] + Wk[4] + Wk[8]) + Wr, \
            [prm.qqr2e * float(Ek.sum()), Ec, El]

    def k2():
        return float((p * p / m1).sum()) / 100.0

    F, W, E = forces(0)
    h, cap = 0.5 * prm.dt, 0.5 * prm.max_disp
    P_ins = 0.0
    for step in range(steps):
        pV += h * ((k2() + W) / (3.0 * L ** 3) - prm.P_ext)
        eps = pV / (3.0 * prm.M_V * L ** 3)
        p = p * math.exp(-eps * h) + 100.0 * F * _expm1_over(-eps * h, h)
        L = (L ** 3 + h * pV / prm.M_V) ** (1.0 / 3.0)
        eps = pV / (3.0 * prm.M_V * L ** 3)
        r = r * math.exp(eps * h) + _cap(p / m1 * _expm1_over(eps * h, h), cap)
        gV, g = math.exp(-prm.gamma_V * prm.dt), math.exp(-prm.gamma * prm.dt)
        pV = pV * gV + math.sqrt(prm.kT * prm.M_V * (1.0 - gV * gV)) * float(_normals(seed, 2, step, np.array([0]))[0][0])
        z = _gpu(np.stack(_normals(seed, 1, step, np.arange(len(m)))[:3], 1))
        p = p * g + torch.sqrt(prm.kT * 100.0 * m1 * (1.0 - g * g)) * z
        eps = pV / (3.0 * prm.M_V * L ** 3)
        r = r * math.exp(eps * h) + _cap(p / m1 * _expm1_over(eps * h, h), cap)
        L = (L ** 3 + h * pV / prm.M_V) ** (1.0 / 3.0)
        r = r - L * torch.floor(r / L)
        F, W, E = forces(step)
        eps = pV / (3.0 * prm.M_V * L ** 3)
        p = p * math.exp(-eps * h) + 100.0 * F * _expm1_over(-eps * h, h)
        P_ins = (k2() + W) / (3.0 * L ** 3)
        pV += h * (P_ins - prm.P_ext)
    cell = np.zeros(32)
    cell[:11] = [L, L, L, pV, W, k2(), P_ins, E[0], E[1], E[2], L ** 3]
    cell[11:12] = np.array([steps], dtype=np.int64).view(np.float64)
    return r, p, F, cell


_PA, _PB = (0, 0, 1), (1, 2, 2)   # the three site pairs of a molecule


def _water(case, seed, key):
    """The rigid-water steps in FP64: tensors of shape (molecules, 3 sites, 3 axes)."""
    pos, mom, q, mass, box, prm = _water_system(case, seed)
    n, alpha, L, pV, wp = case["molecules"], case["alpha"], float(box[0]), 0.0, rbe.water_params()
    q, dd = _gpu(q), _gpu([wp.d_OH ** 2, wp.d_OH ** 2, wp.d_HH ** 2])
    m = _gpu(mass).reshape(n, 3, 1)
    im, M = 1.0 / m, m.sum(1, keepdim=True)
    x, p = _gpu(pos).reshape(n, 3, 3), _gpu(mom).reshape(n, 3, 3)

    def into_box(x):
        return x - L * torch.floor(x[:, :1] / L)

    d = x - x[:, :1]
    x = into_box(x[:, :1] + d - L * torch.round(d / L))
    pairs = _pairs_within(x.reshape(-1, 3), L, prm.rc + 0.3 + 0.15 * case["steps"])
    pairs = pairs[:, pairs[0] // 3 != pairs[1] // 3]
    both_o = (pairs[0] % 3 == 0) & (pairs[1] % 3 == 0)
    sa = math.sqrt(alpha)
    pa, pb = list(_PA), list(_PB)
    D = torch.zeros((3, 3), dtype=torch.float64, device=x.device)   # constraint -> sites, +1 and -1
    for c in range(3):
        D[c, _PA[c]], D[c, _PB[c]] = 1.0, -1.0
    K = torch.einsum("ci,ni,di->ncd", D, im[:, :, 0], D)

    def forces(step):
        r = x.reshape(-1, 3)
        mk, S = _sample([L] * 3, alpha, case["P"], key, step)
        Fk, Wk, Ek = _kspace(r, q, [L] * 3, alpha, mk, S)
        Fr, W, Ec, El = _pair_forces(r, q, L, alpha, prm, pairs, both_o)
        F = (prm.qqr2e * Fk + Fr).reshape(n, 3, 3)
        qm = q.reshape(n, 3)
        s = x[:, pb] - x[:, pa]
        r2 = (s * s).sum(2)
        rr, qq = r2.sqrt(), prm.qqr2e * qm[:, pa] * qm[:, pb]
        ef = torch.special.erf(sa * rr)
        f = qq * (2.0 * sa * torch.exp(-alpha * r2) / (math.sqrt(math.pi) * rr) - ef / r2) / rr
        F = F - torch.einsum("ci,nct->nit", D, f[:, :, None] * s)
        W += float((f * r2).sum()) + prm.qqr2e * float(Wk[0] + Wk[4] + Wk[8])
        R = (m * x).sum(1, keepdim=True) / M
        W -= float((F * (x - R)).sum())
        return F, W, [prm.qqr2e * float(Ek.sum()), Ec, El, -float((qq * ef / rr).sum())]

    def project(p):
        s, v = x[:, pa] - x[:, pb], p * im
        A = K * torch.einsum("nct,ndt->ncd", s, s)
        mu = torch.linalg.solve(A, -((v[:, pa] - v[:, pb]) * s).sum(2, keepdim=True))
        return p + torch.einsum("ci,nct->nit", D, mu * s)

    def kick(p, F, eps):
        Pc, Ft = p.sum(1, keepdim=True), F.sum(1, keepdim=True)
        dP = Pc * math.exp(-eps * h) + 100.0 * Ft * _expm1_over(-eps * h, h) - Pc
        return project(p + 100.0 * h * (F - m * Ft / M) + m / M * dP)

    def drift(x0, p, eps):
        R, Pc = (m * x0).sum(1, keepdim=True) / M, p.sum(1, keepdim=True)
        Rn = R * math.exp(eps * h) + _cap((Pc / M * _expm1_over(eps * h, h))[:, 0], cap)[:, None]
        d = x0 - R
        so = d[:, pa] - d[:, pb]
        dn = d + h * (p * im - Pc / M)
        ds = dn
        for _ in range(8):   # Newton's method on the three multipliers
            s = ds[:, pa] - ds[:, pb]
            g = (s * s).sum(2) - dd
            J = 2.0 * K * torch.einsum("nct,ndt->ncd", s, so)
            ds = ds + im * torch.einsum("ci,nct->nit", D, torch.linalg.solve(J, -g[:, :, None]) * so)
        return Rn + ds, p + m * (ds - dn) / h

    def k2():
        Pc = p.sum(1)
        return float((Pc * Pc / M[:, 0]).sum()) / 100.0

    F, W, E = forces(0)
    h, cap = 0.5 * prm.dt, 0.5 * prm.max_disp
    for step in range(case["steps"]):
        pV += h * ((k2() + W) / (3.0 * L ** 3) - prm.P_ext)
        p = kick(p, F, pV / (3.0 * prm.M_V * L ** 3))
        L = (L ** 3 + h * pV / prm.M_V) ** (1.0 / 3.0)
        x, p = drift(x, p, pV / (3.0 * prm.M_V * L ** 3))
        p = project(p)
        gV, g = math.exp(-prm.gamma_V * prm.dt), math.exp(-prm.gamma * prm.dt)
        pV = pV * gV + math.sqrt(prm.kT * prm.M_V * (1.0 - gV * gV)) * float(_normals(key, 2, step, np.array([0]))[0][0])
        z = _gpu(np.stack(_normals(key, 1, step, np.arange(3 * n))[:3], 1)).reshape(n, 3, 3)
        p = project(p * g + torch.sqrt(prm.kT * 100.0 * m * (1.0 - g * g)) * z)
        x, p = drift(x, p, pV / (3.0 * prm.M_V * L ** 3))
        p = project(p)
        L = (L ** 3 + h * pV / prm.M_V) ** (1.0 / 3.0)
        x = into_box(x)
        F, W, E = forces(step)
        p = kick(p, F, pV / (3.0 * prm.M_V * L ** 3))
        P_ins = (k2() + W) / (3.0 * L ** 3)
        pV += h * (P_ins - prm.P_ext)
    cell = np.zeros(32)
    cell[:11] = [L, L, L, pV, W, k2(), P_ins, E[0], E[1], E[2], L ** 3]
    cell[11:12] = np.array([case["steps"]], dtype=np.int64).view(np.float64)
    cell[25] = E[3]
    return {"pos": x.reshape(-1, 3), "mom": p.reshape(-1, 3), "force": F.reshape(-1, 3), "cell": cell}


def exact(case, seed):
    kind = case["kind"]
    key = 12345 + seed
    if kind == "kspace":
        pos, q, box, alpha = _snapshot(case, seed)
        m, S = _sample(box, alpha, case["P"], key, 3)
        F, W, E = _kspace(_gpu(pos.astype(np.float64)), _gpu(q.astype(np.float64)), box, alpha, m, S)
        return {"forces": F, "virial": W, "energy": E}
    if kind == "batched":
        out = {"forces": [], "virial": [], "energy": []}
        for pos, q, box, sd in _batch_systems(case, seed):
            m, S = _sample(box, 0.2, case["P"], sd, 0)
            F, W, E = _kspace(_gpu(pos), _gpu(q), box, 0.2, m, S)
            for name, v in (("forces", F), ("virial", W[None]), ("energy", E[None])):
                out[name].append(v)
        return {name: torch.cat(v) for name, v in out.items()}
    if kind == "npt":
        pos, mom, q, mass, box = inputs.npt_replica(case["N"], seed)
        r, p, F, cell = _npt(pos, mom, q, mass, box, _npt_params(box, 0.0), 0.2, case["P"], key, case["steps"])
        return {"pos": r, "mom": p, "force": F, "cell": cell}
    if kind == "water":
        return _water(case, seed, key)
    got = [_npt(pos, mom, q, mass, box, prm, 0.2, case["P"], sd, case["steps"])
           for pos, mom, q, mass, box, prm, sd in _serve_requests(case, seed)]
    return {"pos": [g[0] for g in got], "mom": [g[1] for g in got], "cell": [g[3] for g in got]}
