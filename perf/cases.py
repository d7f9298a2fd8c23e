"""Performance cases: the calls that users of the library make, over the sizes, temperatures,
precisions and options that its tests, benchmark and protocol use.

A "step" case advances one lattice (:class:`Lattice`) by MC steps and reads the spins into a
device buffer; "batch" advances replicas together (:class:`Batch`); "static" colours a caller's
own graph (:func:`kw_colour_static`); "full" measures a configuration with the direct sum of the
full Hamiltonian.  ``exact`` recomputes small lattices and the direct sum in numpy / torch.
"""
import math

import numpy as np
import torch

import paper_1503_03295_gb300 as sco

FLOATS = ("e_switched", "e_exchange", "mx", "my", "mz", "m_abs", "m_phi")
WHOLE = ("n_edges", "max_degree", "max_degree_dipolar", "n_colours", "kw_rounds")


def _step(name, Lx, Ly, T, fp64, J=0.0, D=1.0, n_sw=1, sweeps=1, measure=False):
    c = dict(kind="step", Lx=Lx, Ly=Ly, T=T, fp64=fp64, J=J, D=D, n_sw=n_sw, sweeps=sweeps,
             measure=measure)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the parity configuration, measured after every step: the smallest call, all latency
        _step("step_16_fp64", 16, 16, 0.5, True, measure=True),
        # a small ragged lattice of the paper's model (exchange J = 1, D = 0.1), measured
        _step("step_67x41_exchange", 67, 41, 0.85, False, J=1.0, D=0.1, measure=True),
        # the validation lattice of the tests (L = 256) in the FP64 form
        _step("step_256_fp64", 256, 256, 0.6, True),
        # the precision comparison of the benchmark, cold: many pairs survive
        _step("step_1024_fp32", 1024, 1024, 0.4, False),
        # a large ragged lattice, warm, FP64
        _step("step_1000x1337_fp64", 1000, 1337, 0.8, True),
        # the benchmark's lattice in both precisions
        _step("step_2304_fp64", 2304, 2304, 0.6, True),
        _step("step_2304_fp32", 2304, 2304, 0.6, False),
        # one epoch of the paper's schedule: switch and colour once, then 100 MC steps
        _step("epoch_1152_exchange_fp64", 1152, 1152, 0.45, True, J=1.0, D=0.1, n_sw=100,
              sweeps=100),
        # replica sets: 4 sizes x 16 temperatures re-switched every step, and ten runs of the
        # paper's |M_phi|(T) measurement over one epoch
        dict(name="batch_64_replicas", kind="batch", sizes="64,128,256,512", n_T=16, T_lo=0.2,
             T_hi=1.5, fp64=False, J=0.0, D=1.0, n_sw=1, steps=4),
        dict(name="batch_10x128_epoch", kind="batch", sizes="128", n_T=10, T_lo=0.8, T_hi=0.9,
             fp64=False, J=1.0, D=0.1, n_sw=100, steps=100),
        # the allocation-free colouring of a caller's graph
        dict(name="static_400k", kind="static", n=400000, degree=14.0),
        # the full energy of a configuration by direct summation (its largest size)
        dict(name="full_256", kind="full", Lx=256, Ly=256, T=0.6, J=1.0, D=0.1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["epoch", "batch", "static", "full"])
    if kind == "step" or kind == "epoch":
        L = _log(rng, 16, 1800 if kind == "step" else 1000)
        Lx = max(2, int(L * rng.uniform(0.7, 1.3)))
        Ly = max(2, L * L // Lx)
        exchange = kind == "epoch" or rng.random() < 0.3
        T = round(rng.uniform(0.1, 1.25) if exchange else rng.uniform(0.3, 1.5), 3)
        n_sw = 1 if kind == "step" else rng.choice([10, 50, 100])
        return _step(None, Lx, Ly, T, rng.random() < 0.5, J=1.0 if exchange else 0.0,
                     D=0.1 if exchange else 1.0, n_sw=n_sw, sweeps=n_sw, measure=Lx * Ly <= 4096)
    if kind == "batch":
        sizes = ",".join(str(_log(rng, 24, 400)) for _ in range(rng.randint(1, 3)))
        exchange = rng.random() < 0.5
        T_lo = round(rng.uniform(0.25, 0.8), 3)
        return dict(kind="batch", sizes=sizes, n_T=rng.randint(2, 12), T_lo=T_lo,
                    T_hi=round(T_lo + rng.uniform(0.0, 0.6), 3), fp64=rng.random() < 0.3,
                    J=1.0 if exchange else 0.0, D=0.1 if exchange else 1.0,
                    n_sw=10 if exchange else 1, steps=10 if exchange else 4)
    if kind == "static":
        return dict(kind="static", n=_log(rng, 1000, 1 << 20), degree=round(rng.uniform(2.0, 24.0), 2))
    L = _log(rng, 32, 250)
    return dict(kind="full", Lx=L, Ly=_log(rng, 32, 250), T=round(rng.uniform(0.2, 1.5), 3),
                J=rng.choice([0.0, 1.0]), D=rng.choice([0.1, 1.0]))


# ---- what a user holds before the call -----------------------------------------------------
def _stream():
    return torch.cuda.current_stream().cuda_stream


def _params(case, **kw):
    prec = sco.FP64 if case.get("fp64", True) else sco.FP32_GUARDED
    return sco.make_params(case.get("Lx", kw.pop("Lx", None)), case.get("Ly", kw.pop("Ly", None)),
                           J=case["J"], D=case["D"], n_sw=case.get("n_sw", 1), precision=prec,
                           **{"T": case.get("T"), **kw})


def _random_spins(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = torch.randn(3, n, dtype=torch.float64, device="cuda", generator=g)
    return s / s.norm(dim=0)


def _local_graph(n, degree, seed):
    """Symmetric CSR graph with the locality of a switched lattice: vertex i joins i + d, |d| heavy
    tailed (about 1/d^2), or a lattice row (sqrt n) further on; no loops, no double edges."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    m = int(n * degree / 2)
    i = torch.randint(n, (m,), device="cuda", generator=g)
    d = (1.0 / torch.rand(m, device="cuda", dtype=torch.float64, generator=g)).clamp(max=n).long()
    row = max(1, int(math.isqrt(n)))
    j = i + d.clamp(max=n - 1) + row * torch.randint(3, (m,), device="cuda", generator=g)
    keep = j < n
    i, j = i[keep], j[keep]
    key = torch.unique(torch.cat([i * n + j, j * n + i]))
    a, b = key // n, key % n
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(a, minlength=n), 0)
    return rp.to(torch.int32), b.to(torch.int32).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        lat = sco.Lattice(_params(case, seed=seed), stream=_stream())
        return dict(case=case, lat=lat,
                    spins=torch.empty(3, lat.N, dtype=torch.float64, device="cuda"))
    if kind == "batch":
        ps = []
        for a, L in enumerate(int(x) for x in case["sizes"].split(",")):
            for b in range(case["n_T"]):
                T = case["T_lo"] + b * (case["T_hi"] - case["T_lo"]) / max(1, case["n_T"] - 1)
                ps.append(_params(case, Lx=L, Ly=L, T=T, seed=seed * 4096 + a * case["n_T"] + b))
        batch = sco.Batch(ps)
        # a tuning kept from an earlier autotune() of the same kind of set
        batch.set_tuning(steps_per_graph=4, sweep_blocks_per_sm=4, kw_blocks_per_sm=3)
        return dict(case=case, batch=batch, at=np.cumsum([0] + [3 * n for n in batch.N]).tolist(),
                    spins=torch.empty(3 * sum(batch.N), dtype=torch.float64, device="cuda"))
    if kind == "static":
        rp, col = _local_graph(case["n"], case["degree"], seed)
        return dict(case=case, rp=rp, col=col,
                    colour=torch.empty(case["n"], dtype=torch.int32, device="cuda"))
    lat = sco.Lattice(_params(case, seed=seed), stream=_stream())
    spins = _random_spins(lat.N, seed)
    lat.set_spins_device(spins.data_ptr())
    return dict(case=case, lat=lat)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        lat, spins = state["lat"], state["spins"]
        lat.sweep(case["sweeps"])
        lat.get_spins_device(spins.data_ptr())
        if not case["measure"]:
            return [spins]
        o = lat.observables()
        return [spins, [o[k] for k in FLOATS], [o[k] for k in WHOLE]]
    if kind == "batch":
        batch, spins, at = state["batch"], state["spins"], state["at"]
        batch.run(case["steps"])
        for r in range(len(batch)):
            batch.get_spins_device(r, spins.data_ptr() + 8 * at[r])
        return [spins]
    if kind == "static":
        delta, rounds = sco.kw_colour_static(state["rp"].data_ptr(), state["col"].data_ptr(),
                                             case["n"], state["colour"].data_ptr(),
                                             stream=_stream())
        return [state["colour"], delta, rounds]
    o = state["lat"].observables(full=True)
    return [[o[k] for k in FLOATS], o["e_full"]]


# ---- what a pass cannot do without ---------------------------------------------------------
def _survival(lam):
    """Mean of 1 - P over independent uniform spins, lam = beta D / r^3 (an array)."""
    t, w = np.polynomial.legendre.leggauss(24)
    q = np.sqrt(1 + 3 * (0.5 * (t + 1)) ** 2)
    x = lam[:, None] * q
    small = np.minimum(x, 1e-3)
    sh = np.where(x < 1e-3, np.exp(-2 * lam)[:, None] * (1 + small ** 2 / 6),
                  (np.exp(x - 2 * lam[:, None]) - np.exp(-x - 2 * lam[:, None])) / (2 * np.maximum(x, 1e-3)))
    return 1.0 - (sh * (0.5 * w)).sum(1)


def _per_site(bD):
    """Candidates and surviving pair ends per site (bulk, independent spins)."""
    y, x = np.mgrid[0:49, -48:49]
    r2 = (x * x + y * y)[(y > 0) | (x > 0)].astype(float)
    r2 = r2[r2 < 48.0 ** 2]
    lam = bD / r2 ** 1.5
    tail = bD * math.pi / 48.0  # sum of lam beyond r = 48, half plane
    return float((-np.expm1(-4 * lam)).sum() + 4 * tail), 2 * float(_survival(lam).sum() + 2 * tail)


def work(case):
    """Spins read and written once per MC step (48 bytes a site), one operation count per
    candidate of the switch (51) and per pair end of the sweep (120): a pair energy and one or
    two exponentials each.  The colouring reads the graph once."""
    kind = case["kind"]
    if kind in ("step", "batch"):
        if kind == "step":
            reps = [(case["Lx"] * case["Ly"], case["T"])]
            steps = case["sweeps"]
        else:
            T = np.linspace(case["T_lo"], case["T_hi"], case["n_T"])
            reps = [(int(L) ** 2, t) for L in case["sizes"].split(",") for t in T]
            steps = case["steps"]
        flops = bytes_ = 0.0
        for N, T in reps:
            cand, k = _per_site(case["D"] / T)
            flops += N * (51.0 * cand * math.ceil(steps / case["n_sw"]) + 120.0 * k * steps)
            bytes_ += 48.0 * N * steps
        return {"bytes": bytes_, "flops": flops}
    if kind == "static":
        return {"bytes": 4.0 * case["n"] * (2 + case["degree"]), "flops": 0}
    N = case["Lx"] * case["Ly"]
    return {"bytes": 24.0 * N, "flops": 25.0 * N * (N - 1) / 2}


# ---- plain recomputation in 64 bits ----------------------------------------------------------
_M32 = np.uint64(0xFFFFFFFF)


def _mulhilo(a, m):
    m = np.uint64(m)
    al, ah, ml, mh = a & _M32, a >> np.uint64(32), m & _M32, m >> np.uint64(32)
    lo, mid1, mid2 = al * ml, ah * ml, al * mh
    t = (lo >> np.uint64(32)) + (mid1 & _M32) + (mid2 & _M32)
    return ah * mh + (mid1 >> np.uint64(32)) + (mid2 >> np.uint64(32)) + (t >> np.uint64(32)), a * m


def _words(site, step, draw_, tag, seed):
    """Philox4x64-10 of the library's counters (site, step or epoch, draw, tag), key (seed, 0)."""
    c0 = np.asarray(site, np.uint64)
    c1, c2, c3 = (np.broadcast_to(np.asarray(v, np.uint64), c0.shape).copy()
                  for v in (step, draw_, tag))
    k0, k1 = np.uint64(seed), np.uint64(0)
    with np.errstate(over="ignore"):
        for _ in range(10):
            h0, l0 = _mulhilo(c0, 0xD2E7470EE14C6C93)
            h1, l1 = _mulhilo(c2, 0xCA5A826395121157)
            c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
            k0, k1 = k0 + np.uint64(0x9E3779B97F4A7C15), k1 + np.uint64(0xBB67AE8584CAA73B)
    return c0, c1, c2, c3


def _unit(w):
    return (w >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _sphere(n, step, tag, seed):
    """Marsaglia points per site and the third word's uniform of the successful attempt."""
    S, u = np.zeros((n, 3)), np.zeros(n)
    left = np.arange(n)
    for a in range(64):
        w = _words(left, step, a, tag, seed)
        a1, a2 = 2 * _unit(w[0]) - 1, 2 * _unit(w[1]) - 1
        s = a1 * a1 + a2 * a2
        ok = (s > 0) & (s < 1)
        h = np.sqrt(1 - s[ok])
        S[left[ok]] = np.stack([2 * a1[ok] * h, 2 * a2[ok] * h, 1 - 2 * s[ok]], 1)
        u[left[ok]] = _unit(w[2])[ok]
        left = left[~ok]
        if not len(left):
            break
    return S, u


def _table(Lx, Ly):
    y, x = np.mgrid[0:Ly, -(Lx - 1):Lx]
    half = (y > 0) | (x > 0)
    dx, dy = x[half], y[half]
    r2 = dx * dx + dy * dy
    o = np.lexsort((dx, dy, r2))
    dx, dy, r2 = dx[o], dy[o], r2[o]
    q = r2.astype(np.float64)
    A = (2.0 ** 60 / (q * np.sqrt(q)) * (1 + 2.0 ** -50)).astype(np.uint64) + np.uint64(1)
    return dx, dy, q, A


def _energy(D, q, a, b, fx, fy):
    ss = (a * b).sum(-1)
    pa, pb = a[..., 0] * fx + a[..., 1] * fy, b[..., 0] * fx + b[..., 1] * fy
    return D / (q * q * np.sqrt(q)) * (q * ss - 3 * pa * pb)


def _switched(case, S, epoch, seed, tab):
    """Surviving dipolar pairs (i, j, table index) at this epoch."""
    Lx, Ly, D, beta = case["Lx"], case["Ly"], case["D"], 1.0 / case["T"]
    dx, dy, q, A = tab
    W = np.cumsum(A)
    n, K = Lx * Ly, len(A)
    at = np.full(n, -1)
    site = np.arange(n)
    out, t = [], 0
    while len(site):
        w = _words(site, epoch, t // 2, 2, seed)
        up, u = _unit(w[2 * (t % 2)]) + 2.0 ** -53, _unit(w[2 * (t % 2) + 1])
        tau = np.ceil(-np.log(up) / (beta * D) * 2.0 ** 58)
        Ws = np.where(at[site] >= 0, W[np.maximum(at[site], 0)], np.uint64(0))
        room = tau < (W[-1] - Ws).astype(np.float64)
        site, Ws, u = site[room], Ws[room], u[room]
        k = np.maximum(np.searchsorted(W, Ws + tau[room].astype(np.uint64)), at[site] + 1)
        inside = k < K
        site, k, u = site[inside], k[inside], u[inside]
        at[site] = k
        xj, yj = site % Lx + dx[k], site // Lx + dy[k]
        on = (xj >= 0) & (xj < Lx) & (yj < Ly)
        i, kk, uu = site[on], k[on], u[on]
        j = xj[on] + Lx * yj[on]
        vm = D * A[kk].astype(np.float64) * 2.0 ** -59
        V = _energy(D, q[kk], S[i], S[j], dx[kk], dy[kk])
        keep = uu * -np.expm1(-2 * beta * vm) < -np.expm1(beta * (V - vm))
        out.append(np.stack([i[keep], j[keep], kk[keep]]))
        t += 1
    return np.concatenate(out, 1) if out else np.zeros((3, 0), np.int64)


def _colours(nbrs, n):
    """The colouring that halving the palettes group by group from colours v mod g ends in."""
    g = max(len(x) for x in nbrs) + 1
    c = np.arange(n) % g
    G, p, rounds = -(-n // g), 1, 0
    while (1 << (p - 1)) < G:
        grp, right = np.arange(n) // (g << p), (np.arange(n) // (g << (p - 1))) % 2 == 1
        old, rnd, deepest = c.copy(), {}, 0
        for v in sorted(np.flatnonzero(right), key=lambda v: -old[v]):
            used, r = set(), 0
            for u in nbrs[v]:
                if grp[u] != grp[v]:
                    continue
                if not right[u]:
                    used.add(c[u])
                elif old[u] > old[v]:
                    used.add(c[u])
                    r = max(r, rnd[u])
            c[v] = next(x for x in range(g) if x not in used)
            rnd[v] = r + 1
            deepest = max(deepest, r + 1)
        rounds += deepest
        p += 1
    return c, g, rounds


def _exact_step(case, seed):
    Lx, Ly, J, D, beta = case["Lx"], case["Ly"], case["J"], case["D"], 1.0 / case["T"]
    n = Lx * Ly
    tab = _table(Lx, Ly)
    dx, dy, q, A = tab
    S, _ = _sphere(n, 0, 1, seed)
    vm = D * A.astype(np.float64) * 2.0 ** -59
    bonds = [(i, i + 1) for i in range(n) if i % Lx + 1 < Lx] + [(i, i + Lx) for i in range(n - Lx)]
    near = [[] for _ in range(n)]
    for a, b in bonds:
        near[a].append(b)
        near[b].append(a)
    for t in range(case["sweeps"]):
        if t % case["n_sw"] == 0:
            e = _switched(case, S, t // case["n_sw"], seed, tab)
            nb = [set() for _ in range(n)]
            pairs = [[] for _ in range(n)]
            for i, j, k in e.T.tolist():
                nb[i].add(j)
                nb[j].add(i)
                pairs[i].append((j, k))
                pairs[j].append((i, k))
            dip = max(len(x) for x in nb)
            for a, b in bonds if J else ():
                nb[a].add(b)
                nb[b].add(a)
            colour, g, rounds = _colours(nb, n)
        new, u = _sphere(n, t, 3, seed)
        for i in np.argsort(colour, kind="stable"):
            j = np.array([x[0] for x in pairs[i]], int)
            k = np.array([x[1] for x in pairs[i]], int)
            fx, fy = j % Lx - i % Lx, j // Lx - i // Lx
            Vo, Vn = (_energy(D, q[k], s[None, :], S[j], fx, fy) for s in (S[i], new[i]))
            xo, xn = beta * (Vo - vm[k]), beta * (Vn - vm[k])
            dE = (beta * (Vn - Vo) - np.log(-np.expm1(xn)) + np.log(-np.expm1(xo))).sum()
            dE -= beta * J * float((new[i] - S[i]) @ S[near[i]].sum(0)) if near[i] else 0.0
            if u[i] == 0 or math.log(u[i]) + dE < 0:
                S[i] = new[i]
    spins = S.T.copy()
    if not case["measure"]:
        return [spins]
    i, j, k = e
    V = _energy(D, q[k], S[i], S[j], dx[k], dy[k])
    pseudo = (V - np.log(-np.expm1(beta * (V - vm[k]))) / beta).sum()
    ex, site = _exchange_and_moments(torch.from_numpy(spins), Lx, Ly, J)
    return [spins, [pseudo + ex, ex] + site,
            [e.shape[1], g - 1, dip, len(set(colour.tolist())), rounds]]


def _exchange_and_moments(s, Lx, Ly, J):
    n = Lx * Ly
    f = s.reshape(3, Ly, Lx)
    ex = -J * float((f[:, :, 1:] * f[:, :, :-1]).sum() + (f[:, 1:] * f[:, :-1]).sum())
    m = (s.sum(1) / n).tolist()
    ux = torch.arange(Lx, dtype=torch.float64, device=s.device)[None, :] - 0.5 * (Lx - 1)
    uy = torch.arange(Ly, dtype=torch.float64, device=s.device)[:, None] - 0.5 * (Ly - 1)
    r = torch.sqrt(ux * ux + uy * uy)
    phi = torch.where(r > 0, (f[0] * uy - f[1] * ux) / torch.where(r > 0, r, torch.ones_like(r)),
                      torch.zeros_like(r))
    return ex, m + [math.sqrt(sum(x * x for x in m)), float(phi.sum()) / n]


def _exact_full(case, seed):
    """The dipolar sum as a correlation of the zero-padded spin field with each coupling."""
    Lx, Ly, D = case["Lx"], case["Ly"], case["D"]
    s = _random_spins(Lx * Ly, seed)
    f = torch.zeros(3, 2 * Ly, 2 * Lx, dtype=torch.float64, device="cuda")
    f[:, :Ly, :Lx] = s.reshape(3, Ly, Lx)
    F = torch.fft.rfft2(f)
    x = torch.fft.fftfreq(2 * Lx, 1.0 / (2 * Lx), dtype=torch.float64, device="cuda")[None, :]
    y = torch.fft.fftfreq(2 * Ly, 1.0 / (2 * Ly), dtype=torch.float64, device="cuda")[:, None]
    r2 = x * x + y * y
    r2[0, 0] = 1.0
    c3, c5 = r2 ** -1.5, r2 ** -2.5
    c3[0, 0] = c5[0, 0] = 0.0
    pairs = {(0, 0): c3 - 3 * x * x * c5, (1, 1): c3 - 3 * y * y * c5, (2, 2): c3,
             (0, 1): -6 * x * y * c5}
    e = 0.0
    for (a, b), kern in pairs.items():
        h = torch.fft.irfft2(F[b] * torch.fft.rfft2(kern), s=(2 * Ly, 2 * Lx))
        e += 0.5 * float((f[a] * h).sum())
    ex, site = _exchange_and_moments(s, Lx, Ly, case["J"])
    return [[ex, ex] + site, D * e + ex]


def exact(case, seed):
    if case["kind"] == "step" and case["Lx"] * case["Ly"] * case["sweeps"] <= 6000:
        return _exact_step(case, seed)
    if case["kind"] == "full":
        return _exact_full(case, seed)
    return None  # a trajectory that takes minutes here; whole numbers (the colouring)
