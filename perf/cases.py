"""The calls whose speed counts: force evaluations, time steps, the surrogate and
its training, each as a user's program makes it through
``paper_2510_21230_gb300.atm3`` with the state in device memory.

All systems are LJ + ATM fluids in reduced units, r_c = 2.5 and nu = 0.073 (the
workloads of ``synth.py`` and of ``bench.py``), on jittered fcc lattices with
Maxwell-Boltzmann velocities.  FP64 results are handed on in float64, FP32C and
surrogate results in float32, the accuracy those paths state (2e-5 of a force
component); counts are whole numbers.

``exact`` evaluates the same sums in float64 with torch alone: linked-cell
forward lists, every pair of a list, the triplet sum of the energy in r^2 form.
"""
import math

import numpy as np
import torch

from paper_2510_21230_gb300 import atm3, synth

RC, NU, DT = 2.5, 0.073, 0.002
# largest molecule counts drawn
SIZES = {"pair_fp32c": 256000, "pair_fp64": 64000, "product_fp32c": 37000,
         "product_fp64": 24000, "steps_fp32c": 200000, "steps_fp64": 12000}


# ------------------------------------------------------------------ the cases

def _forces(name, n, rho, trav, trunc, prec, aspect=1.0, jitter=0.05, det=False, api="context",
            parts=False):
    return dict(kind="forces", name=name, n=n, rho=rho, aspect=aspect, jitter=jitter, trav=trav,
                trunc=trunc, prec=prec, det=det, api=api, parts=parts)


def _steps(name, n, rho, trav, prec, steps, temperature=1.0, aspect=1.0, graph=False):
    return dict(kind="steps", name=name, n=n, rho=rho, T=temperature, aspect=aspect, trav=trav,
                prec=prec, steps=steps, graph=graph)


def listed():
    return [
        # the smallest liquid of the test suite, the exact path: launches and latency
        _forces("liquid_1k_3c01_fp64", 1000, 0.8, "3c01", "pair", "fp64"),
        # a plug-in that owns the device memory: the call that allocates nothing,
        # a ragged molecule count in a box of three different edges
        _forces("plugin_5k_3c08_fp32c", 5003, 0.6, "3c08", "pair", "fp32c", aspect=1.12,
                api="noalloc"),
        # exact forces of a mid-size liquid: reference and training targets
        _forces("liquid_32k_3c08_fp64", 32000, 0.8, "3c08", "pair", "fp64", parts=True),
        # the product cutoff, the other truncation of every traversal
        _forces("liquid_32k_3c18_product_fp32c", 32000, 0.8, "3c18", "product", "fp32c",
                parts=True),
        # the same in FP64 on the runtime workload's density (odd count)
        _forces("fluid_15k_3c08_product_fp64", 15001, 0.7, "3c08", "product", "fp64",
                parts=True),
        # bitwise repeatable forces of a large ragged system
        _forces("fluid_100k_3c18_det_fp32c", 100003, 0.7, "3c18", "pair", "fp32c", aspect=0.9,
                det=True),
        # the single-phase replay: two small FP64 replicas in one context, ten
        # graph steps, a sample (scalars, pair histogram) and the thermostat
        dict(kind="replay", name="replay_2x1k_fp64", n=1270, n2=1596, rho=0.65, rho2=0.817,
             T=1.033, T2=0.746, trav="3c08", trunc="pair", steps=10),
        # vapour-liquid slab: uneven cells, a density profile after every step
        dict(kind="slab", name="slab_21k_fp32c", edge=30.0, length=120.0, rho=0.73, trav="3c08",
             prec="fp32c", steps=5, bins=600),
        # an ensemble of 64 uneven replicas, autotuned, in graph steps
        dict(kind="batch", name="batch_64_fp32c", count=64, n_lo=500, n_hi=20000, trav="3c08",
             prec="fp32c", steps=4),
        # the headline workload: velocity-Verlet steps of 256,000 molecules
        _steps("liquid_256k_3c08_fp32c", 256000, 0.8, "3c08", "fp32c", 5),
        # learned forces of the same liquid
        dict(kind="surrogate", name="surrogate_256k", n=256000, rho=0.8),
        # training of the learned forces: Adam steps on minibatches
        dict(kind="train", name="train_8k", rows=40000, batch=8192, steps=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges; a product-rule system has six cells or
    more per axis (where cell shifts and minimum image agree)."""
    kind = rng.choice(["forces"] * 6 + ["steps"] * 3 + ["batch", "surrogate", "train", "replay"])
    if kind == "forces":
        prec = rng.choice(["fp64", "fp32c", "fp32c"])
        trunc = rng.choice(["pair", "pair", "product"])
        trav = rng.choice(["3c01", "3c18", "3c08", "3c08", "3c08a"])
        hi = SIZES["%s_%s" % (trunc, prec)]
        if trunc == "product" and trav == "3c01":
            hi //= 2
        n = _log_int(rng, 4000 if trunc == "product" else 500, hi)
        det = trunc == "pair" and rng.random() < 0.25
        api = "noalloc" if n <= 30000 and not det and rng.random() < 0.25 else "context"
        rho = rng.uniform(0.5, 0.85) if trunc == "product" else rng.uniform(0.1, 0.85)
        return _forces("", n, rho, trav, trunc, prec, aspect=rng.uniform(0.92, 1.08),
                       jitter=rng.uniform(0.03, 0.08), det=det, api=api,
                       parts=api == "context" and rng.random() < 0.5)
    if kind == "steps":
        prec = rng.choice(["fp64", "fp32c", "fp32c"])
        return _steps("", _log_int(rng, 1000, SIZES["steps_" + prec]), rng.uniform(0.3, 0.85),
                      rng.choice(["3c18", "3c08", "3c08"]), prec, rng.randint(2, 5),
                      temperature=rng.uniform(0.7, 1.3), aspect=rng.uniform(0.92, 1.08),
                      graph=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind="batch", name="", count=rng.randint(4, 64), n_lo=500,
                    n_hi=_log_int(rng, 2000, 18000), trav=rng.choice(["3c18", "3c08"]),
                    prec="fp32c", steps=rng.randint(2, 4))
    if kind == "surrogate":
        return dict(kind="surrogate", name="", n=_log_int(rng, 1000, 250000),
                    rho=rng.uniform(0.6, 0.85))
    if kind == "train":
        return dict(kind="train", name="", rows=_log_int(rng, 10000, 40000),
                    batch=_log_int(rng, 500, 8192), steps=rng.randint(20, 50))
    return dict(kind="replay", name="", n=_log_int(rng, 1100, 1400), n2=_log_int(rng, 1400, 2400),
                rho=rng.uniform(0.6, 0.7), rho2=rng.uniform(0.75, 0.85), T=1.033, T2=0.746,
                trav=rng.choice(["3c01", "3c18", "3c08"]),
                trunc="pair", steps=rng.randint(5, 10))


# ------------------------------------------------------------------ the inputs

def _fluid(n, rho, temperature, rng, aspect=1.0, jitter=0.05):
    """fcc start in a box of edges (aspect, 1, 1 / aspect) (n / rho)^(1/3)."""
    edge = (n / rho) ** (1.0 / 3.0)
    box = edge * np.array([aspect, 1.0, 1.0 / aspect])
    x = synth.fcc_positions(n, edge, rng, jitter=jitter) * (box / edge)[:, None]
    return dict(n=n, box=box, x=np.ascontiguousarray(x), v=synth.maxwell_boltzmann(n, temperature, rng),
                T=temperature)


def _systems(case, seed):
    """The replicas of a case, host arrays, from the seed alone."""
    rng = np.random.default_rng(seed)
    k = case["kind"]
    if k == "forces":
        return [_fluid(case["n"], case["rho"], 1.0, rng, case["aspect"], case["jitter"])]
    if k == "steps":
        return [_fluid(case["n"], case["rho"], case["T"], rng, case["aspect"])]
    if k == "replay":
        return [_fluid(case["n"], case["rho"], case["T"], rng),
                _fluid(case["n2"], case["rho2"], case["T2"], rng)]
    if k == "slab":
        return [synth.slab(box=(case["edge"], case["edge"], case["length"]), rho_l=case["rho"],
                           seed=seed)]
    if k == "batch":
        # the ensemble's states are the case's; its positions and velocities the seed's
        sizes = np.random.default_rng(case["count"])
        return [_fluid(_log_int(sizes, case["n_lo"], case["n_hi"]), sizes.uniform(0.1, 0.85),
                       sizes.uniform(0.7, 1.3), rng) for _ in range(case["count"])]
    return [_fluid(case["n"], case["rho"], 1.0, rng)]


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _context(systems):
    if len(systems) == 1:
        return atm3.AtmSystem(systems[0]["box"], systems[0]["n"], rc=RC, nu=NU, dt=DT,
                              stream=_stream())
    return atm3.AtmSystem([s["box"] for s in systems], [s["n"] for s in systems], rc=RC, nu=NU,
                          dt=DT, stream=_stream())


def _model(rho, seed):
    """Surrogate weights, and the descriptor statistics of a small liquid."""
    rng = np.random.default_rng(seed)
    s = _fluid(1372, rho, 1.0, rng)
    D, _ = _descriptors(torch.from_numpy(s["x"].T.copy()), s["box"])
    D = D.numpy()
    return (synth.sur_params(seed), D.mean(axis=0).astype(np.float32),
            np.maximum(D.std(axis=0), 1e-3 * np.abs(D).max(axis=0)).astype(np.float32))


def prepare(case, seed):
    if case["kind"] == "train":
        s = atm3.AtmSystem(11.0, 1000, rc=RC, nu=NU, stream=_stream())
        D, V, T = synth.sur_rows(case["rows"], seed)
        s.surrogate_add_rows(D, V, T)
        model = (synth.sur_params(seed + 1), np.zeros(32, np.float32), np.ones(32, np.float32))
        s.surrogate_set_model(*model)
        return dict(case=case, sys=s, model=model, seed=seed)
    systems = _systems(case, seed)
    n = sum(s["n"] for s in systems)
    x = torch.from_numpy(np.concatenate([s["x"] for s in systems], axis=1)).cuda()
    v = torch.from_numpy(np.concatenate([s["v"] for s in systems], axis=1)).cuda()
    state = dict(case=case, x=x, v=v, f=torch.zeros_like(x), f2=torch.zeros_like(x),
                 box=systems[0]["box"], T=[s["T"] for s in systems])
    if case.get("api") == "noalloc":
        return state
    s = state["sys"] = _context(systems)
    if case["kind"] == "forces" and case["det"]:
        s.set_deterministic(True)
    if case["kind"] in ("steps", "slab", "batch", "replay"):
        state["host"] = [torch.empty((3, n), dtype=torch.float64, pin_memory=True)
                         for _ in range(2)]
        if case["kind"] != "slab":
            s.set_options(graph=bool(case.get("graph", True)))
        if case["kind"] == "batch":
            s.set_state(x, v)
            s.build_cells()
            s.autotune(case["trav"], "pair", case["prec"], reps=2)
    if case["kind"] == "surrogate":
        s.surrogate_set_model(*_model(case["rho"], seed))
    return state


# ------------------------------------------------------------------ one pass

def _handed_on(t, prec):
    return t if prec == "fp64" else t.float()


def _frame(state, prec):
    """The new state and its force, as a program stores a frame."""
    s, host = state["sys"], state["host"]
    s.get_forces("total", out=state["f"])
    s.get_state(host[0].numpy(), host[1].numpy())
    x, v = (h.clone() if prec == "fp64" else h.float() for h in host)
    return dict(force=_handed_on(state["f"], prec), x=x, v=v)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        s = state["sys"]
        s.surrogate_set_model(*state["model"])
        loss = s.surrogate_train(case["steps"], batch=case["batch"], lr=1e-3, seed=state["seed"])
        return dict(loss=loss, params=s.surrogate_get_model()[0])
    if kind == "forces":
        prec = case["prec"]
        if case["api"] == "noalloc":
            res = atm3.compute_forces_noalloc(state["box"], state["x"], state["f"], case["trav"],
                                              case["trunc"], prec, rc=RC, nu=NU, stream=_stream())
            return dict(scalars=res, force=_handed_on(state["f"], prec))
        s = state["sys"]
        s.set_state(state["x"])
        s.build_cells()
        res = s.compute_forces(case["trav"], case["trunc"], prec)
        if not case["parts"]:
            s.get_forces("total", out=state["f"])
            return dict(scalars=res, force=_handed_on(state["f"], prec))
        s.get_forces("lj", out=state["f"])
        s.get_forces("atm", out=state["f2"])
        return dict(scalars=res, lj=_handed_on(state["f"], prec), atm=_handed_on(state["f2"], prec))
    s = state["sys"]
    s.set_state(state["x"], state["v"])
    if kind == "surrogate":
        s.build_cells()
        res = s.compute_forces("3c08", "pair", "surrogate")
        s.get_forces("lj", out=state["f"])
        s.get_forces("atm", out=state["f2"])
        return dict(scalars=res, lj=state["f"].float(), atm=state["f2"].float())
    if kind == "replay":
        s.rdf_reset()
        s.step(case["steps"], case["trav"], case["trunc"], "fp64")
        res = s.results()
        s.rdf_accumulate(RC, 250)
        counts, samples = s.rdf_get(250)
        s.get_forces("total", out=state["f"])
        s.thermostat(state["T"])
        s.get_state(state["host"][0].numpy(), state["host"][1].numpy())
        return dict(scalars=res, rdf=counts.astype(np.int64), force=state["f"],
                    x=state["host"][0].clone(), v=state["host"][1].clone())
    prec = case["prec"]
    if kind == "slab":
        s.density_reset()
        for _ in range(case["steps"]):
            s.step(1, case["trav"], "pair", prec, sync=False)
            s.density_accumulate(axis=2, nbins=case["bins"])
        counts, samples = s.density_get(case["bins"])
        return dict(scalars=s.results(), profile=counts.astype(np.int64), **_frame(state, prec))
    s.step(case["steps"], case["trav"], "pair", prec)
    return dict(scalars=s.results() if kind == "steps" else _columns(s.results()),
                **_frame(state, prec))


def _columns(results):
    """The replicas' scalars, an array for each."""
    return {k: np.array([r[k] for r in results],
                        dtype=np.float32 if isinstance(results[0][k], float) else np.int64)
            for k in results[0]}


# ------------------------------------------------------------------ floors

def work(case):
    """Positions (and velocities) in, forces (and the new state) out, once a
    pass; a pair costs 20 flops, a triplet 70 (one squared side from the two
    vectors at its first molecule, the three derivatives, three force terms).
    The triplets of a molecule: rho^2 V^2 15/32 / 6 under the pair rule (V the
    cutoff sphere), about 1800 rho^2 under the product rule."""
    if case["kind"] == "train":
        weights = 32 * 64 + 64 * 64 + 64 * 16
        rows = float(case["steps"]) * case["batch"]
        return dict(bytes=rows * 83 * 4, flops=rows * 6 * weights)
    if case["kind"] == "batch":
        mean_n = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        shape = [(case["count"] * mean_n, 0.475, 0.272)]
    elif case["kind"] == "slab":
        liquid = case["rho"] * case["edge"] ** 2 * 30.0
        shape = [(liquid, case["rho"], case["rho"] ** 2)]
    elif case["kind"] == "replay":
        shape = [(case["n"], case["rho"], case["rho"] ** 2),
                 (case["n2"], case["rho2"], case["rho2"] ** 2)]
    else:
        shape = [(case["n"], case["rho"], case["rho"] ** 2)]
    sphere = 4.0 / 3.0 * math.pi * RC ** 3
    n = sum(s[0] for s in shape)
    pairs = sum(s[0] * s[1] * sphere / 2 for s in shape)
    per = 1800.0 if case.get("trunc") == "product" else sphere ** 2 * 15 / 32 / 6
    triplets = sum(s[0] * s[2] * per for s in shape)
    if case["kind"] == "surrogate":
        mlp = 2.0 * (32 * 64 + 64 * 64 + 64 * 16)
        return dict(bytes=n * 72.0, flops=2 * pairs * 150 + n * mlp)
    steps = case.get("steps", 1)
    return dict(bytes=n * (48.0 if case["kind"] == "forces" else 120.0),
                flops=steps * (20 * pairs + 70 * triplets))


# ------------------------------------------------------------------ 64-bit values

def _forward(x, box, reach=None, whole=False):
    """Padded lists of every molecule's partners in linked cells: later molecules
    of its own cell and those of the 13 forward cells (whole: of all 27).
    Returns index [n, K], displacement [n, K, 3], cell offset [n, K, 3] and
    squared distance [n, K] (infinite where the list has ended); reach: only
    partners closer than that."""
    dev, n = x.device, x.shape[0]
    L = torch.as_tensor(np.asarray(box, dtype=np.float64), device=dev)
    nc = [int(math.floor(float(b) / RC)) for b in box]
    m = torch.tensor(nc, device=dev)
    t = x - torch.floor(x / L) * L
    c = torch.minimum((t / (L / m)).long(), m - 1)
    cid = (c[:, 2] * nc[1] + c[:, 1]) * nc[0] + c[:, 0]
    order = torch.argsort(cid, stable=True)
    count = torch.bincount(cid, minlength=nc[0] * nc[1] * nc[2])
    start = torch.cumsum(count, 0) - count
    place = torch.empty_like(order)
    place[order] = torch.arange(n, device=dev)
    table = torch.full((count.numel(), int(count.max())), -1, device=dev, dtype=torch.long)
    table[cid[order], torch.arange(n, device=dev) - start[cid[order]]] = order
    rows, cols, disp, off = [], [], [], []
    for q in range(0 if whole else 13, 27):
        o = torch.tensor([q % 3 - 1, (q // 3) % 3 - 1, q // 9 - 1], device=dev)
        raw = c + o
        wrap = torch.div(raw, m, rounding_mode="floor")
        nb = raw - wrap * m
        cand = table[(nb[:, 2] * nc[1] + nb[:, 1]) * nc[0] + nb[:, 0]]
        ok = cand >= 0
        if q == 13:
            me = torch.arange(n, device=dev)[:, None]
            ok &= (cand != me) if whole else (place[cand] > place[:, None])
        i, k = ok.nonzero(as_tuple=True)
        j = cand[i, k]
        d = t[j] - t[i] + wrap[i] * L
        if reach is not None:
            near = (d * d).sum(1) < reach * reach
            i, j, d = i[near], j[near], d[near]
        rows.append(i)
        cols.append(j)
        disp.append(d)
        off.append(o.to(torch.int8).expand(i.numel(), 3))
    i, j, d, o = (torch.cat(v) for v in (rows, cols, disp, off))
    by = torch.argsort(i, stable=True)
    i, j, d, o = i[by], j[by], d[by], o[by]
    per = torch.bincount(i, minlength=n)
    slot = torch.arange(i.numel(), device=dev) - (torch.cumsum(per, 0) - per)[i]
    K = max(2, int(per.max()))
    idx = torch.zeros((n, K), device=dev, dtype=torch.long)
    dd = torch.zeros((n, K, 3), device=dev, dtype=torch.float64)
    oo = torch.zeros((n, K, 3), device=dev, dtype=torch.int8)
    r2 = torch.full((n, K), math.inf, device=dev, dtype=torch.float64)
    idx[i, slot], dd[i, slot], oo[i, slot], r2[i, slot] = j, d, o, (d * d).sum(1)
    return idx, dd, oo, r2


def _atm(a, b, c):
    """Energy of Eq. atm in r^2 form and its derivatives by the squared sides."""
    A, B, C = b + c - a, a + c - b, a + b - c
    q2 = 1.0 / (a * b * c)
    q3 = q2 * torch.sqrt(q2)
    P = A * B * C * q2
    u = NU * q3 * (1.0 + 0.375 * P)
    k, q5 = 1.5 + 0.9375 * P, NU * q3 * q2
    return (u, q5 * (0.375 * (2 * a * A - B * C) - k * b * c),
            q5 * (0.375 * (2 * b * B - A * C) - k * a * c),
            q5 * (0.375 * (2 * c * C - A * B) - k * a * b))


def _exact_forces(x, box, trav, trunc):
    """LJ and ATM force [n, 3] and the scalars of one system, in float64."""
    n = x.shape[0]
    flj, fatm = torch.zeros_like(x), torch.zeros_like(x)
    idx, d, off, r2 = _forward(x, box, reach=RC)
    i, k = torch.isfinite(r2).nonzero(as_tuple=True)
    dij, ir2 = d[i, k], 1.0 / r2[i, k]
    s3 = ir2 ** 3
    fw = (48.0 * s3 * s3 - 24.0 * s3) * ir2
    flj.index_add_(0, i, -fw[:, None] * dij)
    flj.index_add_(0, idx[i, k], fw[:, None] * dij)
    e2, w2 = float((4.0 * (s3 * s3 - s3)).sum()), float((fw / ir2).sum())
    owner = trav == "3c01" and trunc == "product"
    if trunc == "product":
        idx, d, off, r2 = _forward(x, box, whole=owner)
    if trav == "3c08a":
        r2 = torch.where((off >= 0).all(2), r2, math.inf)
    K = idx.shape[1]
    jj, kk = torch.triu_indices(K, K, 1, device=x.device)
    e3 = w3 = 0.0
    chunk = max(1, int(1.2e7 / max(1, jj.numel())))
    for m0 in range(0, n, chunk):
        D, R = d[m0:m0 + chunk], r2[m0:m0 + chunk]
        a, b = R[:, jj], R[:, kk]
        c = sum((D[:, :, q][:, kk] - D[:, :, q][:, jj]) ** 2 for q in range(3))
        keep = torch.isfinite(a) & torch.isfinite(b)
        keep &= (c < RC * RC) if trunc == "pair" else (a * b * c < RC ** 6)
        if trav == "3c08" and trunc == "product":
            o = off[m0:m0 + chunk]
            keep &= ((o[:, jj] - o[:, kk]).abs() <= 1).all(2)
        mi, p = keep.nonzero(as_tuple=True)
        a, b, c = a[mi, p], b[mi, p], c[mi, p]
        u, ua, ub, uc = _atm(a, b, c)
        e3 += float(u.sum())
        w3 -= float((2.0 * (ua * a + ub * b + uc * c)).sum())
        dj, dk = D[mi, jj[p]], D[mi, kk[p]]
        fj, fk = 2.0 * ua[:, None] * dj, 2.0 * ub[:, None] * dk
        fatm.index_add_(0, mi + m0, fj + fk)
        if not owner:
            fjk = 2.0 * uc[:, None] * (dk - dj)
            fatm.index_add_(0, idx[mi + m0, jj[p]], fjk - fj)
            fatm.index_add_(0, idx[mi + m0, kk[p]], -fjk - fk)
    if owner:
        e3, w3 = e3 / 3.0, w3 / 3.0
    return flj, fatm, dict(e2=e2, e3=e3, w2=w2, w3=w3)


def _descriptors(x, box):
    """The surrogate's 32 descriptors and 16 vectors [n, 16, 3], in float64."""
    n = x.shape[0]
    idx, d, _, r2 = _forward(x, box, reach=RC)
    i, k = torch.isfinite(r2).nonzero(as_tuple=True)
    j, dij = idx[i, k], d[i, k]
    i, j, dij = torch.cat([i, j]), torch.cat([j, i]), torch.cat([dij, -dij])
    r = dij.norm(dim=1)
    u, fc = dij / r[:, None], 0.5 * (torch.cos(math.pi * r / RC) + 1.0)

    def total(v):
        return torch.zeros((n,) + v.shape[1:], dtype=x.dtype, device=x.device).index_add_(0, i, v)

    dg, dv = (RC - 0.8) / 15, (RC - 0.8) / 4
    D = [total(torch.exp(-(r - 0.8 - q * dg) ** 2 / (2 * dg * dg)) * fc) for q in range(16)]
    p, T = [], []
    eye = torch.eye(3, dtype=x.dtype, device=x.device) / 3.0
    for a in range(4):
        phi = torch.exp(-(r - 0.8 - (a + 0.5) * dv) ** 2 / (2 * dv * dv)) * fc
        p.append(total(phi[:, None] * u))
        if a < 3:
            T.append(total(phi[:, None, None] * (u[:, :, None] * u[:, None, :] - eye)))
    D += [(p[a] * p[b]).sum(1) for a in range(4) for b in range(a, 4)]
    D += [(T[a] * T[b]).sum((1, 2)) for a in range(3) for b in range(a, 3)]
    vec = p + [torch.einsum("nij,nj->ni", T[a], p[b]) for a in range(3) for b in range(4)]
    return torch.stack(D, 1), torch.stack(vec, 1)


def _nothing(keys):
    return {k: None for k in keys}


COUNTS = ("n_cand3", "n_int3", "n_cand2", "n_int2")


def _scalars(e, v=None):
    return dict(e, ekin=None if v is None else float(0.5 * (v * v).sum()), **_nothing(COUNTS))


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return None
    systems = _systems(case, seed)
    dev = _device()
    xs = [torch.from_numpy(s["x"].T.copy()).to(dev) for s in systems]
    if kind == "forces":
        if case["trunc"] == "product" and min(systems[0]["box"]) < 6 * RC:
            return None
        flj, fatm, e = _exact_forces(xs[0], systems[0]["box"], case["trav"], case["trunc"])
        if case["parts"]:
            return dict(scalars=_scalars(e), lj=flj.T.contiguous(), atm=fatm.T.contiguous())
        return dict(scalars=_scalars(e), force=(flj + fatm).T.contiguous())
    if kind == "surrogate":
        flj, _, e = _exact_forces(xs[0], systems[0]["box"], "3c08", "pair")
        P, mean, scale = (torch.from_numpy(np.asarray(w, dtype=np.float64)).to(dev)
                          for w in _model(case["rho"], seed))
        D, vec = _descriptors(xs[0], systems[0]["box"])
        h, at = (D - mean) / scale, 0
        for rows, cols, last in ((32, 64, False), (64, 64, False), (64, 16, True)):
            w = P[at:at + rows * cols].reshape(rows, cols)
            at += rows * cols
            h = h @ w + P[at:at + cols]
            at += cols
            h = h if last else h * torch.sigmoid(h)
        return dict(scalars=dict(_scalars(e), e3=None, w3=None), lj=flj.T.contiguous(),
                    atm=torch.einsum("nm,nmd->dn", h, vec).contiguous())
    trunc = case.get("trunc", "pair")
    out = []
    for s, x in zip(systems, xs):
        L = torch.as_tensor(np.asarray(s["box"], dtype=np.float64), device=dev)
        v = torch.from_numpy(s["v"].T.copy()).to(dev)
        flj, fatm, e = _exact_forces(x, s["box"], case["trav"], trunc)
        for _ in range(case["steps"]):
            v = v + 0.5 * DT * (flj + fatm)
            x = x + DT * v
            x = x - torch.floor(x / L) * L
            flj, fatm, e = _exact_forces(x, s["box"], case["trav"], trunc)
            v = v + 0.5 * DT * (flj + fatm)
        scalars = _scalars(e, v)
        if kind == "replay":
            v = v * math.sqrt(s["T"] * (3 * s["n"] - 3) / (2.0 * scalars["ekin"]))
        out.append((scalars, flj + fatm, x, v))
    force, x, v = (torch.cat([o[q] for o in out]).T.contiguous() for q in (1, 2, 3))
    got = dict(force=force, x=x, v=v)
    if kind == "replay":
        return dict(scalars=[o[0] for o in out], rdf=None, **got)
    if kind == "slab":
        return dict(scalars=[o[0] for o in out], profile=None, **got)
    if kind == "batch":
        return dict(scalars={k: None if k in COUNTS else np.array([o[0][k] for o in out])
                             for k in out[0][0]}, **got)
    return dict(scalars=[o[0] for o in out], **got)
