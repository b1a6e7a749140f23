"""Workloads of the filter library as its users run them, for timing and comparison.

Every case goes through `paper_2509_16896_gb300.binding`, as a user's program does.  The kinds:

  run      one new trajectory through an existing filter: nodes and prior weights
           (`init_nodes`), then K steps on the device (`run_steps`, or one replay of a
           captured CUDA graph); returns the history of the estimates and a checkpoint.
  online   the same trajectory step by step, the estimate read back at every step before the
           next increment is taken (a controller in the loop); the same outputs.
  predict  the prediction alone, from the weights a restart leaves; returns the predicted
           log-weights.
  batch    many ragged filters advanced together.

Sizes are those of the repository's named workloads, its tests and its benchmark, and sizes
between them.  `exact` restates the same numbers in 64-bit torch, without the library.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2509_16896_gb300 import binding

DEV = "cuda:0"
DT = 0.01
NOISE = dict(u=0.7, u_kappa=0.8, u_zero=0, v=1.3, v_kappa=0.5)


def _case(kind, model="cubic", r=0, n=0, N=2, prec="bf16", screen="bf16", R=0.3, interval=2, ess=0.5, K=0,
          graph=False, learned=False, noise=False, materialise=0, members=0, name=None):
    c = dict(kind=kind, model=model, r=r, n=n, N=N, prec=prec, screen=screen, R=R, interval=interval, ess=ess, K=K,
             graph=graph, learned=learned, noise=noise, materialise=materialise, members=members)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a low-dimensional filter in double precision with one global box, in a control loop:
        # the smallest calls, latency and launches only
        _case("online", r=2, n=1024, prec="f64", R=4.0, interval=0, ess=0.0, K=10, name="online_f64_r2_n1024"),
        # mid dimension with the learned restart proposal, in a control loop
        _case("online", r=50, n=8192, K=4, learned=True, name="online_learned_r50_n8192"),
        # the r = 100 workload, throughput mode: a captured graph of steps per trajectory
        _case("run", r=100, n=16384, K=8, graph=True, name="run_bf16_r100_n16384"),
        # the large workload (r = 1000, three bandwidths, e4m3 screen) in throughput mode
        _case("run", r=1000, n=65536, N=3, screen="fp8", K=8, graph=True, name="run_fp8_r1000_n65536"),
        # its dominant layer alone
        _case("predict", r=1000, n=65536, N=3, screen="fp8", name="predict_fp8_r1000_n65536"),
        # the paper's large-scale test: coupled drift, far-off cubic sensor, plain float32 form
        _case("run", model="paper_e1", r=1000, n=2000, prec="f32", ess=0.0, K=8, name="run_e1_f32_r1000_n2000"),
        # the plain float32 prediction (low and mid dimension, or as the accuracy reference)
        _case("predict", r=100, n=16384, prec="f32", name="predict_f32_r100_n16384"),
        # ragged sizes on the plain form: the linear-Gaussian model at low dimension
        _case("predict", model="linear", r=17, n=9001, N=1, prec="f32", name="predict_f32_linear_r17_n9001"),
        # the float32 screen (no tensor cores) in high dimension
        _case("predict", r=1000, n=16384, N=3, prec="f32s", name="predict_f32s_r1000_n16384"),
        # state-dependent noise coefficients
        _case("run", r=40, n=4096, prec="f32", K=6, noise=True, name="run_noise_f32_r40_n4096"),
        # the paper's offline operator, rebuilt at each restart and applied three times
        _case("run", r=100, n=16384, prec="f32", interval=3, ess=0.0, K=3, materialise=2,
              name="run_operator_r100_n16384"),
        # many independent ragged filters (r in 10..200, n in 2048..32768), tuned as a server does
        _case("batch", K=2, members=24, name="batch_24_ragged"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    fam = rng.choice(["high", "mid", "f64", "plain", "plain", "e1", "f32s", "noise", "operator", "batch"])
    if fam == "high":
        r = log_int(100, 1000)
        n = log_int(2048, 65536)
        kind = rng.choice(["run", "predict", "online"])
        return _case(kind, r=r, n=n, N=rng.choice([2, 3]), screen="fp8" if r >= 300 else "bf16",
                     model=rng.choice(["cubic", "linear"]) if r < 300 else "cubic", K=rng.randint(2, 4),
                     graph=(kind == "run"))
    if fam == "mid":
        return _case("online", r=log_int(20, 99), n=log_int(1024, 8192), K=rng.randint(2, 4),
                     learned=rng.random() < 0.5)
    if fam == "f64":
        return _case("online", r=rng.randint(1, 8), n=log_int(256, 2048), N=rng.choice([1, 2]), prec="f64", R=2.0,
                     interval=0, ess=0.0, K=rng.randint(4, 10), model=rng.choice(["cubic", "linear"]))
    if fam == "plain":
        r = log_int(8, 300)
        n = log_int(300, min(16384.0, math.sqrt(2.6e10 / r)))
        return _case("predict", r=r, n=n, N=rng.choice([1, 2, 3]), prec="f32", model=rng.choice(["cubic", "linear"]))
    if fam == "e1":
        return _case("run", model="paper_e1", r=log_int(10, 1000), n=log_int(100, 2000), prec="f32", ess=0.0,
                     K=rng.randint(2, 8))
    if fam == "f32s":
        return _case("predict", r=log_int(100, 1000), n=log_int(1024, 16384), N=rng.choice([2, 3]), prec="f32s")
    if fam == "noise":
        return _case("run", r=log_int(3, 64), n=log_int(512, 4096), prec="f32", K=rng.randint(2, 6), noise=True)
    if fam == "operator":
        return _case("run", r=log_int(20, 100), n=log_int(1024, 16384), prec="f32", interval=3, ess=0.0, K=3,
                     materialise=2)
    return _case("batch", K=rng.randint(1, 2), members=rng.randint(6, 20))


# ---- inputs -----------------------------------------------------------------------------

def _rng(seed, salt):
    return np.random.Generator(np.random.Philox(key=[int(seed) & 0xFFFFFFFFFFFF, salt]))


@functools.lru_cache(maxsize=None)
def _primitive_polynomials(count):
    """The first `count` primitive polynomials over GF(2) as (degree, inner coefficients)."""
    out, deg = [], 1
    while len(out) < count:
        order = (1 << deg) - 1
        primes, v, p = [], order, 2
        while p * p <= v:
            if v % p == 0:
                primes.append(p)
                while v % p == 0:
                    v //= p
            p += 1
        if v > 1:
            primes.append(v)

        def x_to(e, poly):   # x^e modulo poly
            acc, base = 1, 2
            while e:
                if e & 1:
                    acc = mul(acc, base, poly)
                base = mul(base, base, poly)
                e >>= 1
            return acc

        def mul(a, b, poly):
            res = 0
            while b:
                if b & 1:
                    res ^= a
                b >>= 1
                a <<= 1
                if (a >> deg) & 1:
                    a ^= poly
            return res

        for a in range(1 << (deg - 1)):
            poly = (1 << deg) | (a << 1) | 1
            if deg == 1 or (x_to(order, poly) == 1 and all(x_to(order // q, poly) != 1 for q in primes)):
                out.append((deg, a))
                if len(out) == count:
                    break
        deg += 1
    return out


def _sobol_tables(r, seed):
    """Generator parameters and scramble draws in the layout of `init_nodes`."""
    g = _rng(seed, 11)
    poly = np.zeros((r, binding.SOBOL_POLY_WORDS), dtype=np.uint32)
    deg = np.zeros(r, dtype=np.int64)
    for d, (s, a) in enumerate(_primitive_polynomials(r - 1) if r > 1 else [], start=1):
        poly[d, 0], poly[d, 1], deg[d] = s, a, s
    draws = g.random((r, 14))
    for k in range(1, 15):   # m_k odd, below 2^k
        m = 2 * np.floor(draws[:, k - 1] * (1 << (k - 1))).astype(np.uint32) + 1
        poly[:, 1 + k] = np.where(deg >= k, m, 0) if 1 + k < binding.SOBOL_POLY_WORDS else 0
    raw = g.integers(0, 1 << 32, size=(r, 33), dtype=np.uint64)
    scr = np.zeros((r, binding.SOBOL_SCRAMBLE_WORDS), dtype=np.uint32)
    for k in range(1, 33):
        above = np.uint64(((1 << 32) - 1) ^ ((1 << (33 - k)) - 1))
        scr[:, k - 1] = ((raw[:, k - 1] & above) | np.uint64(1 << (32 - k))).astype(np.uint32)
    scr[:, 32] = raw[:, 32].astype(np.uint32)
    return poly, scr


def _increments(case, r, K, model, seed):
    """Observation increments of one simulated trajectory (Euler--Maruyama, x_0 ~ N(0, I))."""
    g = _rng(seed, 23)
    x = g.standard_normal(r)
    out = np.empty((K, r))
    for k in range(K):
        if model == "cubic":
            f = np.cos(x)
        elif model == "linear":
            f = -0.5 * x
        else:
            xn = np.concatenate([x[1:], [0.0]])
            f = np.sin(x) * (-0.5 * x + 0.1 * xn) + np.sin(2 * x) * (-0.3 * x + 0.3 * xn)
        su = NOISE["u"] * (1 + NOISE["u_kappa"] * np.sin(x) ** 2) if case["noise"] else 1.0
        x = x + DT * f + math.sqrt(DT) * su * g.standard_normal(r)
        h = x ** 3 if model == "cubic" else (x if model == "linear" else (x - 100.0) ** 3)
        sv = NOISE["v"] * (1 + NOISE["v_kappa"] * np.sin(x) ** 2) if case["noise"] else 1.0
        out[k] = h * DT + math.sqrt(DT) * sv * g.standard_normal(r)
    return out


def _restart_state(r, R, seed):
    """Centre and per-coordinate variance at a restart: the estimate of a tracked state, most
    variances under the floor (R / 4)^2, some above it."""
    g = _rng(seed, 37)
    centre = g.standard_normal(r)
    var = (R / 4) ** 2 * np.maximum(1.0, g.uniform(0.0, 1.6, r))
    return centre, var


def _members(case, seed):
    """Sizes of a ragged batch (the same for every seed: a server's fleet) and their models."""
    g = _rng(case["members"], 41)
    out = []
    for b in range(case["members"]):
        r = int(g.integers(10, 201))
        n = int(round(math.exp(g.uniform(math.log(2048.0), math.log(32768.0)))))
        out.append(dict(case, r=r, n=n, model="cubic" if b % 2 == 0 else "linear", seed=seed * 1000 + b))
    return out


def _config(c):
    return binding.make_config(model=c["model"], r=c["r"], n=c["n"], dt=DT, R=c["R"], n_scales=c["N"],
                               precision=c["prec"], restart_interval=c["interval"], ess_frac=c["ess"],
                               restart_rule="learned" if c["learned"] else "plain", screen_type=c["screen"],
                               noise=NOISE if c["noise"] else None, materialise=c["materialise"])


def _network_params(r, hidden, seed):
    g = _rng(seed, 53)
    shapes = [(hidden, 3 * r), (hidden,), (hidden, hidden), (hidden,), (2 * r, hidden), (2 * r,)]
    return np.concatenate([(g.standard_normal(s) / math.sqrt(s[-1]) * (0.05 if i == 4 else 1.0)
                            if len(s) == 2 else np.zeros(s)).ravel()
                           for i, s in enumerate(shapes)]).astype(np.float32)


def _log_weights(u, mask, var):
    """Log-weights a restart leaves at nodes u (offsets from the new centre), normalised."""
    lw = -0.5 * (u.double() ** 2 / torch.tensor(var, device=u.device)).sum(1)
    lw[mask] = -math.inf
    return lw - torch.logsumexp(lw, 0)


def prepare(case, seed):
    torch.cuda.set_device(DEV)
    if case["kind"] == "batch":
        mem = _members(case, seed)
        bt = binding.Batch([_config(m) for m in mem], device=DEV)
        for b, m in enumerate(mem):
            poly, scr = _sobol_tables(m["r"], m["seed"])
            centre, var = _restart_state(m["r"], m["R"], m["seed"])
            u = _nodes(m["r"], m["n"], m["R"], m["seed"])
            bt.filters[b].init_nodes(poly, scr, centre)
            bt.filters[b].set_state(centre, _log_weights(u, _mask(u, m["R"]), var).float().cpu().numpy(), 0.0, 1)
        bt.autotune(None, reps=2)
        dy = np.concatenate([_increments(case, m["r"], case["K"], m["model"], m["seed"]) for m in mem], axis=1)
        return dict(case=case, batch=bt, dys=torch.tensor(dy, dtype=torch.float64, device=DEV),
                    hist=torch.zeros((case["K"], bt.H), dtype=torch.float64, device=DEV),
                    fields=[torch.tensor(i, device=DEV) for i in _batch_fields(mem)])
    r, n = case["r"], case["n"]
    poly, scr = _sobol_tables(r, seed)
    flt = binding.Filter(_config(case), device=DEV, stream=torch.cuda.Stream(DEV))
    st = dict(case=case, flt=flt, poly=poly, scr=scr, centre=np.zeros(r))
    if case["kind"] == "predict":
        centre, var = _restart_state(r, case["R"], seed)
        flt.init_nodes(poly, scr, centre)
        u = _nodes(r, n, case["R"], seed)
        flt.set_state(centre, _log_weights(u, _mask(u, case["R"]), var).float().cpu().numpy(), 0.0, 1)
        for _ in range(12 if case["prec"] == "bf16" else 1):   # a running filter has settled its screen
            flt.predict()
        flt.get_log_weights()
        return st
    st["dys"] = torch.tensor(_increments(case, r, case["K"], case["model"], seed), dtype=torch.float64, device=DEV)
    if case["learned"]:
        st["net"] = binding.MLP(r, 256, max_batch=8, device=DEV, stream=flt.stream)
        st["net"].set_params(_network_params(r, 256, 5))
        flt.set_restart_mlp(st["net"])
    flt.init_nodes(poly, scr, st["centre"])
    if case["kind"] == "run":
        st["hist"] = torch.zeros((case["K"], 2 * r + 4), dtype=torch.float64, device=DEV)
        if case["graph"]:
            torch.cuda.synchronize()
            flt.graph_capture(st["dys"], st["hist"])
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        bt = state["batch"]
        bt.run_steps(state["dys"], state["hist"])
        return [state["hist"][:, i] for i in state["fields"]]
    flt = state["flt"]
    if kind == "predict":
        flt.predict()
        return flt.get_log_weights()
    flt.init_nodes(state["poly"], state["scr"], state["centre"])
    if kind == "online":
        out = []
        for k in range(case["K"]):
            flt.predict()
            flt.update(state["dys"][k])
            out.append(flt.estimate())
            flt.restart()
        return out, _checkpoint(flt)
    if case["graph"]:
        flt.graph_launch()
    else:
        flt.run_steps(state["dys"], state["hist"])
    return _history(state["hist"], flt.r), _checkpoint(flt)


def _history(h, r):
    """The rows' fields: estimate, variance, and ESS, Lambda, Z, restart flag each."""
    return [h[:, :r], h[:, r:2 * r]] + [h[:, 2 * r + i] for i in range(4)]


def _batch_fields(mem):
    """Columns of a batch's history row per field: all members' estimates, variances, ..."""
    cols, o = [[] for _ in range(6)], 0
    for m in mem:
        r = m["r"]
        cols[0] += range(o, o + r)
        cols[1] += range(o + r, o + 2 * r)
        for i in range(4):
            cols[2 + i].append(o + 2 * r + i)
        o += 2 * r + 4
    return cols


def _checkpoint(flt):
    """What a user saves to resume: box centre, running normaliser, step, log-weights."""
    centre, z, k = flt.get_state()
    return centre, z, k, flt.get_log_weights()[0]


# ---- work of one pass ----------------------------------------------------------------------

def work(case):
    """Bytes: the nodes written once (a new trajectory) and read once per step, weights and
    increments in, estimates out.  Operations: per step the update (about 20 per coordinate of
    a node) and, for the forms that evaluate every pair, the squared distance and the drift
    product of every pair (subtract, two multiply-adds counted as in the benchmark: 3 n^2 r).
    A screened prediction has no such floor: it proves pairs negligible without them."""
    if case["kind"] == "batch":
        parts = [_work_one(dict(m, kind="steps")) for m in _members(case, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    return _work_one(case)


def _work_one(c):
    r, n = float(c["r"]), float(c["n"])
    K = 1 if c["kind"] == "predict" else c["K"]
    ub = 4.0 * n * r
    by = K * ub + 8.0 * n * K + 8.0 * K * (3 * r + 4)
    fl = 0.0
    if c["kind"] != "predict":
        fl += 20.0 * n * r * K
    if c["kind"] in ("run", "online"):
        by += ub
    if c["prec"] in ("f32", "f64"):
        fl += 3.0 * n * n * r * (1 if c["materialise"] else K)
        if c["materialise"]:
            by += (1 + K) * 4.0 * c["N"] * n * n
    return {"bytes": by, "flops": fl}


# ---- the same numbers in 64 bits --------------------------------------------------------------

def _nodes(r, n, R, seed):
    """float32 box coordinates [n][r] of the scrambled Sobol points (device)."""
    poly, scr = _sobol_tables(r, seed)
    V = np.zeros((33, r), dtype=np.int64)
    s = poly[:, 0].astype(np.int64)
    a = poly[:, 1].astype(np.int64)
    for k in range(1, 33):
        init = poly[:, min(1 + k, binding.SOBOL_POLY_WORDS - 1)].astype(np.int64) << (32 - k)
        rec = np.zeros(r, dtype=np.int64)
        for sd in np.unique(s[(s > 0) & (s < k)]):
            sel = s == sd
            v = V[k - sd, sel] ^ (V[k - sd, sel] >> sd)
            for i in range(1, sd):
                v ^= np.where((a[sel] >> (sd - 1 - i)) & 1, V[k - i, sel], 0)
            rec[sel] = v
        V[k] = np.where(s == 0, 1 << (32 - k), np.where(s >= k, init, rec)) & 0xFFFFFFFF
    W = np.zeros((33, r), dtype=np.int64)   # scrambled: digit k is the parity of row k
    for k in range(1, 33):
        x = V[1:] & scr[:, k - 1].astype(np.int64)
        for sh in (16, 8, 4, 2, 1):
            x ^= x >> sh
        W[1:] |= (x & 1) << (32 - k)
    W = torch.tensor(W, device=DEV)
    idx = torch.arange(n, device=DEV)
    gray = idx ^ (idx >> 1)
    y = torch.tensor(scr[:, 32].astype(np.int64), device=DEV).expand(n, r).clone()
    for b in range(max(1, int(n - 1).bit_length())):
        y ^= ((gray >> b) & 1)[:, None] * W[b + 1][None, :]
    t = (y.double() + 0.5) * 2.0 ** -31 - 1.0
    return (R * t).float()


def _mask(u, R):
    return (u.double().abs() >= R - 1e-12 * R).any(1)


def _coefficients(N):
    A = np.zeros((N + 1, N + 1))
    A[0] = 1.0
    rhs = np.zeros(N + 1)
    rhs[0] = rhs[1] = 1.0
    for j in range(N):
        A[1, j] = 2.0 ** -j
        for k in range(N - 1):
            A[2 + k, j] = 2.0 ** (-j * (1.5 + 0.5 * k))
    c = np.linalg.solve(A, rhs)
    if N == 1:
        c[1] = 0.0
    return c


def _drift64(c, x):
    if c["model"] == "cubic":
        return torch.cos(x), -torch.sin(x).sum(1)
    if c["model"] == "linear":
        return -0.5 * x, torch.full((x.shape[0],), -0.5 * x.shape[1], dtype=x.dtype, device=x.device)
    xn = torch.cat([x[:, 1:], torch.zeros_like(x[:, :1])], 1)
    ax, bx = -0.5 * x + 0.1 * xn, -0.3 * x + 0.3 * xn
    s1, c1, s2, c2 = torch.sin(x), torch.cos(x), torch.sin(2 * x), torch.cos(2 * x)
    return s1 * ax + s2 * bx, (c1 * ax - 0.5 * s1 + 2 * c2 * bx - 0.3 * s2).sum(1)


def _predict64(c, u, centre, logw, mask):
    """Predicted log-weights relative to the largest kernel offset, and that offset."""
    r, n, N = c["r"], c["n"], c["N"]
    taus = [DT / 2 ** j for j in range(N)]
    lwq = r * math.log(2 * c["R"]) - math.log(n)
    C = [-0.5 * r * math.log(2 * math.pi * t) + lwq for t in taus]
    cref = max(C)
    coef = _coefficients(N)
    src = logw.masked_fill(mask, -math.inf)
    usq = (u * u).sum(1)
    pred = torch.empty(n, dtype=torch.float64, device=u.device)
    step = max(1, int(1.5e8 // n))
    for a in range(0, n, step):
        ut = u[a:a + step]
        x = centre + ut
        f, div = _drift64(c, x)
        hld = 0.0
        if c["noise"]:
            U = NOISE["u"] * (1 + NOISE["u_kappa"] * torch.sin(x) ** 2)
            m = 1.0 / U ** 2
            hld = torch.log(U).sum(1)
            S1 = (m * ut * ut).sum(1, keepdim=True) + m @ (u * u).T - 2 * (m * ut) @ u.T
        else:
            m = torch.ones_like(ut)
            S1 = (ut * ut).sum(1, keepdim=True) + usq[None, :] - 2 * ut @ u.T
        mf = m * f
        S2 = (mf * ut).sum(1, keepdim=True) - mf @ u.T
        nf = (mf * f).sum(1)
        terms = []
        for j, t in enumerate(taus):
            L = torch.logsumexp(S2 - S1 / (2 * t) + src[None, :], 1) - 0.5 * t * nf
            terms.append(math.log(abs(coef[j])) + C[j] - cref - t * div - hld + L)
        signs = [math.copysign(1.0, v) for v in coef[:N]]
        if coef[N] != 0.0:
            terms.append(math.log(abs(coef[N])) + logw[a:a + step] - cref)
            signs.append(math.copysign(1.0, coef[N]))
        terms = torch.stack(terms, 1)
        top = terms.max(1).values
        tot = (torch.tensor(signs, dtype=torch.float64, device=u.device) *
               torch.exp(terms - top[:, None])).nan_to_num(0.0).sum(1)
        pred[a:a + step] = torch.where(tot > 0, top + torch.log(tot.clamp_min(1e-300)),
                                       torch.full_like(top, -math.inf))
    return pred.masked_fill(mask, -math.inf), cref


def _steps64(c, u, centre, logw, dys, step0=0):
    """K filter steps: rows of (mean, variance, ESS, Lambda, Z, restart), and the state after
    them (centre, Z, step, log-weights)."""
    r, n = c["r"], c["n"]
    mask = _mask(u, c["R"])
    u = u.double()
    Z, rows = 0.0, []
    for k in range(dys.shape[0]):
        pred, cref = _predict64(c, u, centre, logw, mask)
        x = centre + u
        h = x ** 3 if c["model"] == "cubic" else (x if c["model"] == "linear" else (x - 100.0) ** 3)
        if c["noise"]:
            ib = (NOISE["v"] * (1 + NOISE["v_kappa"] * torch.sin(x) ** 2)) ** -2
            ll = (ib * (h * dys[k] - 0.5 * DT * h * h)).sum(1)
        else:
            ll = (h * dys[k] - 0.5 * DT * h * h).sum(1)
        upd = pred + ll
        lam = torch.logsumexp(upd, 0)
        logw = upd - lam
        lam = float(lam) + cref
        Z += lam
        w = torch.exp(logw)
        off = w @ u
        mean = centre + off
        var = w @ (u - off) ** 2
        ess = float(1.0 / (w * w).sum())
        kk = step0 + k + 1
        due = (c["ess"] > 0 and ess < c["ess"] * n) or (c["interval"] >= 2 and kk % c["interval"] == 0)
        rows.append((mean, var, ess, lam, Z, 1.0 if due else 0.0))
        if due:
            centre = mean
            v = torch.clamp(var, min=(c["R"] / 4) ** 2)
            lw = (-0.5 * u * u / v).sum(1).masked_fill(mask, -math.inf)
            logw = lw - torch.logsumexp(lw, 0)
    return rows, (centre.cpu().numpy(), Z, step0 + dys.shape[0], logw.cpu().numpy())


def _hist64(rows):
    h = torch.stack([torch.cat([m, v, torch.tensor([e, l, z, d], dtype=torch.float64, device=m.device)])
                     for m, v, e, l, z, d in rows])
    return _history(h, rows[0][0].shape[0])


def exact(case, seed):
    kind = case["kind"]
    if case["learned"]:   # the network's products take 16-bit operands by design
        return None
    if kind == "batch":
        cols = []
        for m in _members(case, seed):
            u = _nodes(m["r"], m["n"], m["R"], m["seed"])
            centre, var = _restart_state(m["r"], m["R"], m["seed"])
            lw = _log_weights(u, _mask(u, m["R"]), var).float().double()
            dy = torch.tensor(_increments(case, m["r"], case["K"], m["model"], m["seed"]), device=DEV)
            cols.append(_hist64(_steps64(m, u, torch.tensor(centre, device=DEV), lw, dy, 1)[0]))
        return [torch.cat([f if f.dim() == 2 else f[:, None] for f in fs], 1) for fs in zip(*cols)]
    r, n, R = case["r"], case["n"], case["R"]
    if float(n) * n * r * max(1, case["K"]) > 2.5e12:   # tens of seconds of 64-bit products
        return None
    u = _nodes(r, n, R, seed)
    mask = _mask(u, R)
    if kind == "predict":
        centre, var = _restart_state(r, R, seed)
        lw = _log_weights(u, mask, var).float().double()
        pred, cref = _predict64(case, u.double(), torch.tensor(centre, device=DEV), lw, mask)
        return pred.cpu().numpy(), cref
    centre = torch.zeros(r, dtype=torch.float64, device=DEV)
    lw = (-0.5 * u.double() ** 2).sum(1).masked_fill(mask, -math.inf)
    lw = lw - torch.logsumexp(lw, 0)
    dys = torch.tensor(_increments(case, r, case["K"], case["model"], seed), device=DEV)
    rows, end = _steps64(case, u, centre, lw, dys)
    if kind == "online":
        return [(m.cpu().numpy(), v.cpu().numpy(), e, z) for m, v, e, _, z, _ in rows], end
    return _hist64(rows), end
