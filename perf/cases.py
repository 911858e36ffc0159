"""The calls whose speed counts: one problem, many problems, points, optimal
transport and the differentiable loss, each through the package's public
functions at the sizes of the paper's experiments and of this repository's
benchmark and tests.

listed() gives the fixed cases, draw(rng) one more of the same ranges,
prepare(case, seed) the inputs on the GPU, run(state) one call, work(case) the
bytes and operations a call cannot do without, and exact(case, seed) the
outputs in plain torch, 64 bits wide.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2203_03732_gb300 as prot

DEV = "cuda"


def listed():
    return [
        # a small assignment inside a host program that needs the answer (and
        # the phase counts) at once: launches and latency are all there is
        dict(name="assign_n300_sync", kind="assign", rows=300, cols=300, dtype="float64", squared=False,
             eps=0.1, rule="lowest", host=False, sync=True),
        # the repository's first workload: 1000 points, squared distances
        dict(name="assign_n1000", kind="assign", rows=1000, cols=1000, dtype="float64", squared=True,
             eps=0.1, rule="lowest", host=False, sync=False),
        # the paper's synthetic experiment at its largest size: the benchmark's headline
        dict(name="assign_n10000", kind="assign", rows=10000, cols=10000, dtype="float64", squared=False,
             eps=0.01, rule="lowest", host=False, sync=False),
        # the same experiment at its coarsest eps, costs in 32 bits: one phase of many rounds
        dict(name="assign_n10000_coarse_f32", kind="assign", rows=10000, cols=10000, dtype="float32",
             squared=False, eps=0.1, rule="lowest", host=False, sync=False),
        # sides of different size, rows that start on no 16-byte boundary
        dict(name="assign_2999x4507_f32", kind="assign", rows=2999, cols=4507, dtype="float32", squared=False,
             eps=0.02, rule="lowest", host=False, sync=False),
        # a fine guarantee (floor(1/eps) > 252): rounded costs of 16 bits, thousands of short rounds
        dict(name="assign_n1000_fine", kind="assign", rows=1000, cols=1000, dtype="float64", squared=False,
             eps=0.003, rule="lowest", host=False, sync=False),
        # costs in pinned host memory, results back on the host: the end-to-end call
        dict(name="assign_n10000_host", kind="assign", rows=10000, cols=10000, dtype="float64", squared=False,
             eps=0.01, rule="lowest", host=True, sync=True),
        # the sequential greedy at the paper's finest eps, where it is the fastest rule
        dict(name="assign_n10000_sequential", kind="assign", rows=10000, cols=10000, dtype="float64",
             squared=False, eps=0.005, rule="sequential", host=False, sync=False),
        # points instead of a cost matrix
        dict(name="points_n10000", kind="points", rows=10000, cols=10000, dim=2, squared=False, eps=0.01),
        # many small and middling problems of ragged sizes in one call
        dict(name="batched_512", kind="batched", problems=512, n_min=64, n_max=2048, size_seed=4,
             dtype="float32", eps=0.01),
        # a training step on point clouds: loss and its gradients
        dict(name="loss_64x4096", kind="loss", problems=64, n=4096, dim=3, eps=0.01),
        # optimal transport between weighted point sets
        dict(name="ot_n10000", kind="ot", rows=10000, cols=10000, dtype="float64", eps=0.05),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]; every other one is made odd."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.5:
        n |= 1
    return max(lo, min(hi, n))


def draw(rng):
    kind = rng.choice(["assign", "assign", "assign", "points", "batched", "loss", "ot"])
    dtype = rng.choice(["float32", "float64"])
    if kind == "assign":
        rows = _log_int(rng, 128, 10000)
        cols = rows if rng.random() < 0.6 else min(10000, rows + _log_int(rng, 1, 4000))
        rule = rng.choice(["lowest", "lowest", "lowest", "offset", "sequential"])
        host = rng.random() < 0.2
        # the fine guarantee stays with the sizes at which it takes milliseconds
        eps = rng.choice([0.1, 0.05, 0.02, 0.01] + ([0.003] if rows <= 1000 else []))
        return dict(kind=kind, rows=rows, cols=cols, dtype=dtype, squared=rng.random() < 0.3, eps=eps,
                    rule=rule, host=host, sync=host or rows < 1000)
    if kind == "points":
        rows = _log_int(rng, 128, 10000)
        cols = rows if rng.random() < 0.6 else min(10000, rows + _log_int(rng, 1, 4000))
        return dict(kind=kind, rows=rows, cols=cols, dim=rng.choice([2, 2, 3, 5]),
                    squared=rng.random() < 0.5, eps=rng.choice([0.1, 0.05, 0.02, 0.01]))
    if kind == "batched":
        n_max = _log_int(rng, 64, 2048)
        return dict(kind=kind, problems=_log_int(rng, 8, 512), n_min=max(1, n_max // 32), n_max=n_max,
                    size_seed=rng.randrange(1 << 30), dtype="float32" if n_max > 1024 else dtype,
                    eps=rng.choice([0.1, 0.05, 0.02, 0.01]))
    if kind == "loss":
        return dict(kind=kind, problems=_log_int(rng, 4, 64), n=_log_int(rng, 128, 4096),
                    dim=rng.choice([2, 3]), eps=rng.choice([0.1, 0.05, 0.02, 0.01]))
    return dict(kind=kind, rows=_log_int(rng, 128, 10000), cols=_log_int(rng, 128, 10000), dtype=dtype,
                eps=rng.choice([0.1, 0.05]))


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _sizes(case):
    g = np.random.Generator(np.random.PCG64(case["size_seed"]))
    return [int(n) for n in g.integers(case["n_min"], case["n_max"] + 1, case["problems"])]


def _cost_matrix(XB, XA, squared, out):
    """|b - a|^2 or |b - a| over the largest, rows = B, formed in FP64."""
    for s in range(0, XB.shape[0], 1024):
        acc = None
        for d in range(XB.shape[1]):
            t = XB[s:s + 1024, d, None] - XA[None, :, d]
            acc = t * t if acc is None else acc + t * t
        out[s:s + 1024] = acc if squared else acc.sqrt()
    out /= out.max()
    return out


def _uniform_costs(g, rows, cols, dim, squared, dtype):
    """Points uniform in the unit cube (A drawn before B) and their cost matrix."""
    XA = torch.rand((cols, dim), generator=g, device=DEV, dtype=torch.float64)
    XB = torch.rand((rows, dim), generator=g, device=DEV, dtype=torch.float64)
    C = torch.empty((rows, cols), device=DEV, dtype=getattr(torch, dtype))
    return _cost_matrix(XB, XA, squared, C)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    st = dict(case)
    if kind == "assign":
        C = _uniform_costs(g, case["rows"], case["cols"], 2, case["squared"], case["dtype"])
        if case["host"]:
            H = torch.empty(C.shape, dtype=C.dtype, pin_memory=True)
            H.copy_(C)
            C = H
        st["C"] = C
    elif kind == "points":
        st["XA"] = torch.rand((case["cols"], case["dim"]), generator=g, device=DEV)
        st["XB"] = torch.rand((case["rows"], case["dim"]), generator=g, device=DEV)
    elif kind == "batched":
        n = _sizes(case)
        C = torch.empty(sum(k * k for k in n), device=DEV, dtype=getattr(torch, case["dtype"]))
        off = 0
        for k in n:
            C[off:off + k * k] = _uniform_costs(g, k, k, 3, True, case["dtype"]).reshape(-1)
            off += k * k
        st.update(C=C, sizes=n)
    elif kind == "loss":
        shape = (case["problems"], case["n"], case["dim"])
        st["X"] = torch.randn(shape, generator=g, device=DEV).requires_grad_(True)
        st["Y"] = torch.randn(shape, generator=g, device=DEV).requires_grad_(True)
        st["g"] = torch.rand(case["problems"], generator=g, device=DEV) + 0.5
    else:
        st["C"] = _uniform_costs(g, case["rows"], case["cols"], 2, False, case["dtype"])
        for side, n in (("demand", case["cols"]), ("supply", case["rows"])):
            m = -torch.log1p(-torch.rand(n, generator=g, device=DEV, dtype=torch.float64))  # Dirichlet(1)
            st[side] = m / m.sum()
        # plans hold about 1.5 entries a vertex
        st["plan_cap"] = 8 * (case["rows"] + case["cols"])
        st["slot"] = torch.arange(st["plan_cap"], device=DEV)
    return st


def _counted(res):
    """The solve's result with its phase and round counts in the place of the statistics."""
    stats = res.pop("stats", None)
    if stats is not None:
        res["phases"], res["rounds"] = stats["phases"], stats["rounds"]
    return res


def run(state):
    kind = state["kind"]
    if kind == "assign":
        return _counted(prot.assign(state["C"], state["eps"], rule=state["rule"], sync=state["sync"]))
    if kind == "points":
        return prot.assign_points(state["XA"], state["XB"], state["eps"], sync=False,
                                  metric="sqeuclidean" if state["squared"] else "euclidean")
    if kind == "batched":
        return prot.assign_batched(state["C"], state["sizes"], state["eps"], sync=False)
    if kind == "loss":
        loss = prot.assignment_loss(state["X"], state["Y"], state["eps"])
        gX, gY = torch.autograd.grad(loss, (state["X"], state["Y"]), state["g"])
        return dict(loss=loss.detach(), grad_X=gX, grad_Y=gY)
    res = prot.ot(state["C"], state["supply"], state["demand"], state["eps"], plan_cap=state["plan_cap"], sync=False)
    past = state["slot"] >= res["plan_nnz"]  # a plan of fixed length, empty past its last entry
    for k in ("plan_row", "plan_col", "plan_mass"):
        res[k].masked_fill_(past, 0)
    return res


def work(case):
    """Inputs once and outputs once; one operation per cost that is rounded
    and the operations of a distance where the costs come from points.  (How
    often a rounded cost is looked at again depends on the values.)"""
    kind = case["kind"]
    if kind == "batched":
        n = _sizes(case)
        w = 4 if case["dtype"] == "float32" else 8
        sq, tot = sum(k * k for k in n), sum(n)
        return {"bytes": w * sq + 16 * tot + 16 * len(n), "flops": sq}
    if kind == "loss":
        P, n, d = case["problems"], case["n"], case["dim"]
        return {"bytes": P * (16 * n * d + 8), "flops": P * n * n * (3 * d + 1)}
    rows, cols = case["rows"], case["cols"]
    if kind == "points":
        return {"bytes": 4 * case["dim"] * (rows + cols) + 8 * (rows + cols) + 8,
                "flops": rows * cols * (3 * case["dim"] + 1)}
    w = 4 if case["dtype"] == "float32" else 8
    if kind == "assign":
        return {"bytes": w * rows * cols + 8 * (rows + cols) + 8, "flops": rows * cols}
    return {"bytes": w * rows * cols + 8 * (rows + cols) + 16 * (rows + cols) + 4 * rows + 12 * cols + 8,
            "flops": rows * cols}


# ---------------------------------------------------------------------------
# The outputs in plain torch.
# ---------------------------------------------------------------------------
_NONE = 1 << 30


def _rounded(C, eps):
    """floor(c / eps) of the exact quotient, int16: the IEEE quotient's floor,
    corrected by one where k * eps (split so that each product is exact) is
    above c or (k + 1) * eps is not."""
    hi = float((np.array([eps]).view(np.uint64) & np.uint64(0xFFFFFFFFFC000000)).view(np.float64)[0])
    lo = eps - hi
    out = torch.empty(C.shape, dtype=torch.int16, device=C.device)
    for s in range(0, C.shape[0], 1024):
        c = C[s:s + 1024].double()
        k = torch.floor(c / eps)
        k = k - ((c - k * hi) < k * lo).double()
        k1 = k + 1
        k = k + ((c - k1 * hi) >= k1 * lo).double()
        out[s:s + 1024] = k.to(torch.int16)
    return out


def _first(adm, col):
    """The lowest admissible column of every row, _NONE where there is none."""
    return torch.where(adm, col, _NONE).amin(1)


def _first_cyclic(adm, col, start):
    """The same for a scan that starts at column start[row] and goes round once."""
    turn = torch.where(adm, (col - start[:, None]) % col.numel(), _NONE).amin(1)
    return torch.where(turn == _NONE, turn, (turn + start) % col.numel())


def _seeded_start(phase, nB, nA, device):
    """The offset rule's first column of every row: SplitMix64 of (phase, row) mod n_A."""
    x = (np.uint64(phase) << np.uint64(32)) | np.arange(nB, dtype=np.uint64)
    x = x + np.uint64(0x9E3779B97F4A7C15)
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    x = x ^ (x >> np.uint64(31))
    return torch.from_numpy((x % np.uint64(nA)).astype(np.int32)).to(device)


def _lowest_proposer(cols, rows, n):
    best = torch.full((n,), _NONE, dtype=torch.int32, device=rows.device)
    return best.scatter_reduce_(0, cols.long(), rows.int(), "amin")


def _match_rounds(cb, T, offset=False):
    """Every phase of the main routine with the round rule: each free row
    proposes to its lowest admissible untaken column (with offset: the first
    from its seeded start on), each column takes its lowest proposer.  Returns (mate_row, mate_col, y_row, key, phases, rounds)."""
    nB, nA = cb.shape
    i32 = dict(dtype=torch.int32, device=cb.device)
    y, k = torch.ones(nB, **i32), torch.zeros(nA, dtype=torch.int16, device=cb.device)
    mb, ma = torch.full((nB,), -1, **i32), torch.full((nA,), -1, **i32)
    col = torch.arange(nA, **i32)
    phases = rounds = 0
    while True:
        act = (mb < 0).nonzero()[:, 0]
        if act.numel() <= T:
            return mb, ma, y, k.int(), phases, rounds
        phases += 1
        taken = torch.zeros(nA, dtype=torch.bool, device=cb.device)
        start = _seeded_start(phases, nB, nA, cb.device) if offset else None
        while act.numel():
            f = []
            for r in act.split(2048):
                adm = (cb[r] + k == (y[r] - 1).to(torch.int16)[:, None]) & ~taken
                f.append(_first_cyclic(adm, col, start[r]) if offset else _first(adm, col))
            f = torch.cat(f)
            stuck = f == _NONE
            y[act[stuck]] += 1
            act, f = act[~stuck], f[~stuck].long()
            if act.numel() == 0:
                break
            rounds += 1
            won = _lowest_proposer(f, act, nA)[f] == act
            w, a = act[won], f[won]
            old = ma[a].long()
            mb[old[old >= 0]] = -1
            ma[a], mb[w] = w.int(), a.int()
            taken[a] = True
            act = act[~won]
        k += taken.to(torch.int16)


def _match_greedy(cb, T):
    """The same with the sequential greedy: the free rows in index order."""
    c = cb.cpu().numpy()
    nB, nA = c.shape
    y, k = np.ones(nB, np.int32), np.zeros(nA, np.int16)
    mb, ma = np.full(nB, -1, np.int32), np.full(nA, -1, np.int32)
    phases = 0
    while True:
        free = np.flatnonzero(mb < 0)
        if free.size <= T:
            t = [torch.from_numpy(v).to(cb.device) for v in (mb, ma, y, k.astype(np.int32))]
            return (*t, phases, phases)
        phases += 1
        kk = k.copy()  # a taken column's key is moved out of every target's reach
        for b in free:
            hit = c[b] + kk == y[b] - 1
            a = int(hit.argmax())
            if not hit[a]:
                y[b] += 1
                continue
            kk[a] = 0x3FFF
            k[a] += 1
            if ma[a] >= 0:
                mb[ma[a]] = -1
            ma[a], mb[b] = b, a


def _complete(mb, ma):
    """The k-th free row takes the k-th free column."""
    fb = (mb < 0).nonzero()[:, 0]
    fa = (ma < 0).nonzero()[:fb.numel(), 0]
    mb, ma = mb.clone(), ma.clone()
    mb[fb], ma[fa] = fa.int(), fb.int()
    return mb, ma


def _solved(cb, eps, rule="lowest"):
    T = math.floor(eps * cb.shape[0])
    match = _match_greedy(cb, T) if rule == "sequential" else _match_rounds(cb, T, rule == "offset")
    mb, ma, y, k, phases, rounds = match
    mb, ma = _complete(mb, ma)
    return dict(row_to_col=mb, col_to_row=ma, y_row=y, y_col=-k), phases, rounds


def _dist32(XB, XA, squared):
    """Distances in FP32, one rounded operation at a time, as the points entry defines its costs."""
    acc = None
    for d in range(XB.shape[1]):
        t = XB[:, d, None] - XA[None, :, d]
        acc = t * t if acc is None else acc + t * t
    return acc if squared else acc.sqrt()


def _points_rounded(XB, XA, squared, eps):
    d = _dist32(XB, XA, squared)
    return _rounded(d / d.max(), eps)


def _matched_distance(XB, XA, mate, squared):
    t = ((XB.double() - XA.double()[mate.long()]) ** 2).sum(1)
    return (t if squared else t.sqrt()).sum()


def _ot_clusters(cb, S, D, eps):
    """The cluster phases of the transport form.  Returns (F, kmin, clo, chi,
    matched copies [n_dem][n_sup])."""
    nB, nA = cb.shape
    dev = cb.device
    F, f = torch.ones(nB, dtype=torch.int32, device=dev), S.clone()
    kmin, clo, chi = torch.zeros_like(D), D.clone(), torch.zeros_like(D)
    lo = torch.zeros((nA, nB), dtype=torch.int32, device=dev)
    hi = torch.zeros_like(lo)
    col = torch.arange(nA, dtype=torch.int32, device=dev)
    T = math.floor(eps * int(S.sum()))
    while int(f.sum()) > T:
        r, avail = f.clone(), clo.clone()
        act = (r > 0).nonzero()[:, 0]
        while act.numel():
            k16 = kmin.to(torch.int16)
            p = torch.cat([_first((cb[b] + k16 == (F[b] - 1).to(torch.int16)[:, None]) & (avail > 0), col)
                           for b in act.split(2048)])
            act, p = act[p != _NONE], p[p != _NONE].long()
            if act.numel() == 0:
                break
            best = _lowest_proposer(p, act, nA)
            a = (best != _NONE).nonzero()[:, 0]
            w = best[a].long()
            g = torch.minimum(r[w], avail[a])
            avail[a] -= g
            r[w] -= g
            f[w] -= g
            clo[a] -= g
            chi[a] += g
            for q in (kmin[a] >= 1).nonzero()[:, 0].split(1024):  # evict, highest supply first
                have = lo[a[q]]
                above = have.flip(1).cumsum(1, dtype=torch.int32).flip(1) - have
                take = torch.minimum((g[q][:, None] - above).clamp_min(0), have)
                lo[a[q]] = have - take
                f += take.sum(0, dtype=torch.int32)
            hi[a, w] += g
            act = act[r[act] > 0]
        F[(r > 0)] += 1
        up = (clo == 0) & (chi > 0)
        kmin[up] += 1
        clo[up], chi[up] = chi[up], 0
        lo[up], hi[up] = hi[up], 0
    return F, kmin, clo, chi, lo.add_(hi)


def _ot_cost(C, nu, mu, count, theta):
    """Cost of the plan count / theta after the fix-up (excess returned by the
    highest supplier, the rest routed north-west)."""
    m = count.double() / theta
    excess = (m.sum(1) - mu).clamp_min(0)
    sup = torch.arange(m.shape[1], device=m.device)
    last = torch.where(m > 0, sup, -1).amax(1)
    got = (last >= 0).nonzero()[:, 0]
    m[got, last[got]] -= torch.minimum(excess[got], m[got, last[got]])
    cost = sum((m[:, s:s + 1024] * C[s:s + 1024].double().T).sum() for s in range(0, m.shape[1], 1024))
    P = (nu - m.sum(0)).clamp_min(0).cumsum(0)
    Q = (mu - m.sum(1)).clamp_min(0).cumsum(0)
    ends = torch.cat([P, Q]).clamp_max(torch.minimum(P[-1], Q[-1])).sort().values
    size = ends.diff(prepend=ends.new_zeros(1))
    at = ends - size / 2
    b = torch.searchsorted(P, at).clamp_max(P.numel() - 1)
    a = torch.searchsorted(Q, at).clamp_max(Q.numel() - 1)
    return cost + (size * C[b, a].double()).sum()


def exact(case, seed):
    kind, eps = case["kind"], case["eps"]
    st = prepare(case, seed)
    if kind == "assign":
        C = st["C"].to(DEV)
        out, phases, rounds = _solved(_rounded(C, eps), eps, case["rule"])
        out["cost"] = C.gather(1, out["row_to_col"].long()[:, None]).double().sum()
        if case["sync"]:
            out["phases"], out["rounds"] = phases, rounds
        return {k: v.cpu() if case["host"] and torch.is_tensor(v) else v for k, v in out.items()}
    if kind == "points":
        out, _, _ = _solved(_points_rounded(st["XB"], st["XA"], case["squared"], eps), eps)
        out["cost"] = _matched_distance(st["XB"], st["XA"], out["row_to_col"], case["squared"])
        return out
    if kind == "batched":
        if case["problems"] > 64:  # about 0.2 s a problem at the larger sizes
            return None
        parts, costs, phases, off = [], [], [], 0
        for n in st["sizes"]:
            C = st["C"][off:off + n * n].view(n, n)
            off += n * n
            out, ph, _ = _solved(_rounded(C, eps), eps)
            parts.append(out)
            costs.append(C.gather(1, out["row_to_col"].long()[:, None]).double().sum())
            phases.append(ph)
        res = {k: torch.cat([p[k] for p in parts]) for k in ("row_to_col", "col_to_row", "y_row", "y_col")}
        return dict(res, costs=torch.stack(costs), phases=torch.tensor(phases, dtype=torch.int64, device=DEV))
    if kind == "loss":
        X, Y, g = st["X"].detach(), st["Y"].detach(), st["g"].double()
        n = case["n"]
        loss, gX, gY = [], torch.empty_like(X, dtype=torch.float64), torch.empty_like(Y, dtype=torch.float64)
        for i in range(case["problems"]):
            out, _, _ = _solved(_points_rounded(X[i], Y[i], True, eps), eps)
            mate = out["row_to_col"].long()
            loss.append(_matched_distance(X[i], Y[i], mate, True) / n)
            gX[i] = 2.0 * (X[i].double() - Y[i].double()[mate]) / n * g[i]
            gY[i, mate] = -gX[i]
        return dict(loss=torch.stack(loss), grad_X=gX, grad_Y=gY)
    # transport: which pairs the fix-up adds hangs on the last bit of its
    # residuals, so the plan has no value of its own; its cost has one
    theta = 4.0 * max(case["rows"], case["cols"]) / eps
    S = torch.floor(theta * st["supply"]).int()
    D = torch.ceil(theta * st["demand"]).int()
    F, kmin, clo, chi, count = _ot_clusters(_rounded(st["C"], eps), S, D, eps)
    cost = _ot_cost(st["C"], st["supply"], st["demand"], count, theta)
    return dict(plan_row=None, plan_col=None, plan_mass=None, plan_nnz=None, y_sup=F, dem_kmin=kmin, dem_lo=clo,
                dem_hi=chi, cost=cost)
