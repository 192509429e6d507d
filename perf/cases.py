"""Performance cases of the Schulze library: the work a user's program has it
do, through the package's public calls.

A case is a dict of plain values; ``"call"`` says which call it makes. Ballots
are drawn on the GPU from the seed: full or top-k Mallows rankings around a
random reference order, Plackett-Luce lists with Zipf(1.1) weights (the shape
of streaming-chart data) and weak orders in tiers. Sizes are those of the
repository's workloads and the ranges around them.
"""
import math

import numpy as np
import torch

import paper_2505_12976_gb300 as S

DEV = "cuda"


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # A committee or club ballot: one small election with full rankings,
        # where latency and launches count.
        dict(name="small_full", call="run", model="mallows", m=64, n=1000, k=64, phi=0.8, margin=False),
        # One election of a few hundred candidates, odd sizes, full rankings,
        # with the paper's margin weights.
        dict(name="full_margin", call="run", model="mallows", m=381, n=2777, k=381, phi=0.98, margin=True),
        # A large field of which the voters list their favourites: a few of
        # the candidates get all the votes.
        dict(name="large_topk", call="run", model="mallows", m=4096, n=20000, k=50, phi=0.9, margin=False),
        # The largest profile with every count beyond 16 bits possible:
        # popularity-weighted short lists over many candidates.
        dict(name="huge_pl", call="run", model="zipf", m=16384, n=200000, k=20, phi=0.0, margin=False),
        # A profile shaped like the paper's largest chart data set: long
        # lists, every candidate listed, counts within 16 bits.
        dict(name="spotify_like", call="run", model="zipf", m=18407, n=15553, k=200, phi=0.0, margin=False),
        # A service that receives ballots in (page-locked) host memory and
        # answers with winners and order on the host.
        dict(name="host_topk", call="run_host", model="mallows", m=4096, n=20000, k=50, phi=0.9, margin=False),
        # Ballots with ties: positions in, counts, widths and ranking out by
        # the separate calls.
        dict(name="weak_orders", call="weak", model="mallows", m=1024, n=20000, k=1024, phi=0.97, tier=16),
        # Thousands of uneven small elections in one launch (surveys, polls
        # of many districts): sizes uniform up to the maxima.
        dict(name="batch_mixed", call="batch", E=4096, m_lo=8, m_hi=512, n_lo=50, n_hi=5000),
        # Labelling one training election of the proposal network: the whole
        # path, then the candidates' features.
        dict(name="label_topk", call="label", model="mallows", m=1237, n=9001, k=57, phi=0.9, margin=False),
        # Winners only of a large top-k election by proposal and certificate,
        # with the network's weights.
        dict(name="winners_fast", call="fast", model="mallows", m=8192, n=20000, k=50, phi=0.9, net=True),
        # Winners only of a dense chart-shaped profile, Copeland proposals
        # (too many candidates with edges to certify: the propagation decides).
        dict(name="winners_dense", call="fast", model="zipf", m=18407, n=15553, k=200, phi=0.0, net=False),
        # One training step of the proposal network on 64 elections.
        dict(name="train_step", call="train", elections=64, m_lo=256, m_hi=2048),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["full", "topk", "zipf", "host", "weak", "batch", "label", "fast", "dense", "train"])
    if kind == "full":
        m = _log(rng, 8, 1024)
        return dict(call="run", model="mallows", m=m, n=_log(rng, 50, 20000), k=m,
                    phi=round(rng.uniform(0.6, 1.0), 3), margin=rng.random() < 0.5)
    if kind == "zipf":
        k = rng.randint(10, 200)
        return dict(call="run", model="zipf", m=_log(rng, 512, 16384), n=min(_log(rng, 2000, 200000), 4000000 // k), k=k,
                    phi=0.0, margin=rng.random() < 0.3)
    if kind in ("topk", "host"):
        return dict(call="run" if kind == "topk" else "run_host", model="mallows", m=_log(rng, 256, 4096),
                    n=_log(rng, 1000, 60000), k=rng.randint(10, 100), phi=round(rng.uniform(0.6, 0.99), 3),
                    margin=rng.random() < 0.3)
    if kind == "weak":
        m = _log(rng, 32, 1024)
        return dict(call="weak", model="mallows", m=m, n=_log(rng, 200, 20000), k=m,
                    phi=round(rng.uniform(0.6, 1.0), 3), tier=rng.randint(1, 24))
    if kind == "batch":
        return dict(call="batch", E=_log(rng, 64, 3000), m_lo=8, m_hi=rng.randint(32, 512), n_lo=50,
                    n_hi=_log(rng, 200, 5000))
    if kind == "label":
        return dict(call="label", model="mallows", m=rng.randint(256, 2048), n=rng.randint(1000, 20000),
                    k=rng.randint(10, 100), phi=round(rng.uniform(0.6, 0.99), 3), margin=False)
    if kind == "fast":
        return dict(call="fast", model="mallows", m=_log(rng, 512, 8192), n=_log(rng, 1000, 20000),
                    k=rng.randint(10, 100), phi=round(rng.uniform(0.6, 0.95), 3), net=rng.random() < 0.5)
    if kind == "dense":
        k = rng.randint(50, 200)
        return dict(call="fast", model="zipf", m=_log(rng, 4096, 18407), n=_log(rng, 4000, 15553), k=k, phi=0.0,
                    net=rng.random() < 0.5)
    lo = rng.randint(64, 256)
    return dict(call="train", elections=rng.randint(8, 64), m_lo=lo, m_hi=rng.randint(lo, 2048))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _mallows(g, n, m, k, phi):
    """int32 [n, k]: place t takes the j-th of the remaining candidates of a
    random reference order with probability proportional to phi**j."""
    left = (m - torch.arange(k, device=DEV, dtype=torch.float64))[:, None]
    u = torch.rand((k, n), generator=g, device=DEV, dtype=torch.float64)
    j = torch.floor(u * left) if phi >= 1.0 else torch.floor(torch.log1p(-u * (1.0 - phi ** left)) / math.log(phi))
    code = torch.minimum(j.clamp_(min=0), left - 1).to(torch.int32)
    del u, j
    for t in range(k - 2, -1, -1):  # places among the remaining -> places in the reference order
        rest = code[t + 1:]
        rest += rest >= code[t]
    ref = torch.randperm(m, generator=g, device=DEV, dtype=torch.int32)
    return ref[code.t().contiguous().long()]


def _zipf(g, n, m, k):
    """int32 [n, k]: Plackett-Luce with weight (popularity rank + 1)**-1.1,
    drawn as the k largest of log weight + Gumbel noise."""
    logw = -1.1 * torch.log(torch.arange(1, m + 1, device=DEV, dtype=torch.float32))
    logw = logw[torch.randperm(m, generator=g, device=DEV)]
    out = torch.empty((n, k), dtype=torch.int32, device=DEV)
    step = max(1, (1 << 27) // m)
    for v in range(0, n, step):
        e = torch.empty((min(step, n - v), m), device=DEV).exponential_(generator=g)
        out[v:v + step] = torch.topk(logw - torch.log(e), k, dim=1).indices
    return out


def _ballots(case, g):
    if case["model"] == "zipf":
        return _zipf(g, case["n"], case["m"], min(case["k"], case["m"]))
    return _mallows(g, case["n"], case["m"], min(case["k"], case["m"]), case["phi"])


def _positions(ranks, m, tier=1):
    """[n, m] positions of the candidates on ballots that list k of them."""
    n, k = ranks.shape
    pos = torch.full((n, m), k, dtype=torch.int32, device=DEV)
    place = torch.arange(k, dtype=torch.int32, device=DEV) // tier
    return pos.scatter_(1, ranks.long(), place.expand(n, k).contiguous())


def _batch_sizes(case):
    """Sizes of the case's elections (the same for every seed)."""
    rs = np.random.RandomState(case["E"])
    m = rs.randint(case["m_lo"], case["m_hi"] + 1, case["E"]).astype(np.int32)
    n = rs.randint(case["n_lo"], case["n_hi"] + 1, case["E"]).astype(np.int32)
    return n, m


def _batch_ballots(case, g, seed):
    """Full rankings packed back to back: every second election impartial
    culture, the others concentrated around a random reference order."""
    n, m = _batch_sizes(case)
    spread = np.random.RandomState(int(seed) % (1 << 32)).uniform(0.5, 1.0, case["E"])
    out = torch.empty(int((n.astype(np.int64) * m).sum()), dtype=torch.int32, device=DEV)
    at = 0
    for e in range(case["E"]):
        ne, me = int(n[e]), int(m[e])
        key = torch.empty((ne, me), device=DEV).exponential_(generator=g)
        if e % 2 == 0:  # weights falling geometrically along the reference order
            key *= torch.randperm(me, generator=g, device=DEV).float().mul_(-math.log(spread[e])).clamp_(max=80.0).exp_()
        out[at:at + ne * me] = torch.argsort(key, dim=1).flatten()
        at += ne * me
    return out


def _network(g):
    """Weights whose scores follow wins minus losses, as a trained proposal
    network's do, over small random values elsewhere (16-64-64-1, flat)."""
    w = 1e-4 * torch.randn(S.NPARAM, generator=g, device=DEV)
    w1, w2, w3 = w[0:1024].view(64, 16), w[1088:5184].view(64, 64), w[5248:5312]
    w1[0, 0] += 1.0  # hidden unit 0: the share of wins, unit 1: of losses
    w1[1, 1] += 1.0
    w2[0, 0] += 1.0
    w2[1, 1] += 1.0
    w3[0] += 4.0
    w3[1] -= 4.0
    return w


def _train_inputs(case, g):
    rs = np.random.RandomState(case["elections"])
    sizes = rs.randint(case["m_lo"], case["m_hi"] + 1, case["elections"])
    seg = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    N = int(seg[-1])
    s = torch.rand(N, generator=g, device=DEV)  # a candidate's strength
    e = torch.from_numpy(np.repeat(np.arange(len(sizes)), sizes)).to(DEV)
    best = torch.zeros(len(sizes), device=DEV).scatter_reduce(0, e, s, "amax")
    label = (s >= best[e] - 0.001).to(torch.int32)
    t = torch.rand((N, 16), generator=g, device=DEV) * 0.05
    for q, (a, b) in enumerate([(0, 1), (1, -1), (0, 0), (0.2, 0.6), (0.8, -0.6), (0.1, 0.8), (0.9, -0.8), (0, 0),
                                (-0.8, 1.6), (0, 0.4), (0.4, -0.4), (-0.9, 0.8), (0.1, 0.8), (0.1, 0.8), (1, -1),
                                (1, -1)]):
        t[:, q] += a + b * s
    t[:, 7] = (s < 0.5).float()
    theta = torch.randn(S.NPARAM, generator=g, device=DEV) * 0.15
    theta[1024:1088] = 0
    theta[5184:5248] = 0
    theta[5312] = 0
    m1 = 1e-3 * torch.randn(S.NPARAM, generator=g, device=DEV)
    m2 = 1e-6 * (0.5 + torch.rand(S.NPARAM, generator=g, device=DEV))
    return dict(theta=theta, m1=m1, m2=m2, step=37, feat=t, label=label, seg=torch.from_numpy(seg).to(DEV), lr=3e-3)


# ------------------------------------------------------------------ the calls

def _flags(case):
    return S.F_MARGIN if case.get("margin") else 0


def prepare(case, seed):
    g, call = _gen(seed), case["call"]
    st = dict(case=case)
    if call in ("run", "label"):
        st["ranks"] = _ballots(case, g)
    elif call == "run_host":
        st["ranks"] = _ballots(case, g).cpu().pin_memory()
        st["winners"] = torch.empty(case["m"], dtype=torch.int32).pin_memory()
        st["order"] = torch.empty(case["m"], dtype=torch.int32).pin_memory()
    elif call == "weak":
        st["pos"] = _positions(_ballots(case, g), case["m"], case["tier"])
    elif call == "batch":
        n, m = _batch_sizes(case)
        st["ranks"] = _batch_ballots(case, g, seed)
        st["plan"] = S.SchulzeBatch(n, m, m)
        st["out"] = [torch.empty(st["plan"].vec_elems, dtype=torch.int32, device=DEV) for _ in range(3)]
    elif call == "fast":
        st["d"] = S.schulze_tally(_ballots(case, g), case["m"])
        st["params"] = _network(g) if case["net"] else None
    elif call == "train":
        st.update(_train_inputs(case, g))
    return st


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "run":
        return S.schulze_run(state["ranks"], case["m"], flags=_flags(case))
    if call == "label":
        out = S.schulze_run(state["ranks"], case["m"])
        out["feat"] = S.schulze_features(out["d"], case["n"])
        return out
    if call == "run_host":
        w, o = S.schulze_run_host(state["ranks"], case["m"], flags=_flags(case), winners=state["winners"],
                                  order=state["order"])
        return {"winners": w, "order": o}
    if call == "weak":
        d = S.schulze_tally_positions(state["pos"])
        p = S.schulze_strongest_paths(d, case["n"])
        order, beaten_by = S.schulze_ranking(p)
        return {"d": d, "p": p, "order": order, "beaten_by": beaten_by}
    if call == "batch":
        w, o, b = state["out"]
        state["plan"].run(state["ranks"], winners=w, order=o, beaten_by=b)
        return {"winners": w, "order": o, "beaten_by": b}
    if call == "fast":
        w, stats = S.schulze_winners_fast(state["d"], case["n"], state["params"])
        return {"winners": w, "stats": stats}
    # the step updates its arguments: on copies, so that every pass takes the same step
    theta, m1, m2 = state["theta"].clone(), state["m1"].clone(), state["m2"].clone()
    loss, grad = S.schulze_mlp_train_step(theta, m1, m2, state["step"], state["feat"], state["label"], state["seg"],
                                          state["lr"])
    return {"params": theta, "adam_m": m1, "adam_v": m2, "loss": loss, "grad": grad}


# ------------------------------------------------------------------ the work

def _listed(case):
    """Candidates on some ballot, about (all of them for Zipf lists)."""
    m, n, k = case["m"], case["n"], min(case["k"], case["m"])
    if case["model"] == "zipf" or case["phi"] >= 1.0:
        return m
    return min(m, int(k + math.log(n * k) / -math.log(case["phi"])))


def work(case):
    """Bytes: inputs and outputs once. flops: the pairwise counts (compares of
    full rankings, increments of top-k lists), two per (max, min) update of
    Floyd-Warshall among the listed candidates, the features' statistics and
    the network's multiplies and adds."""
    call = case["call"]
    if call == "batch":
        n, m = (x.astype(np.float64) for x in _batch_sizes(case))
        return {"bytes": float((4 * n * m + 12 * m).sum()), "flops": float((n * m * m / 2 + 2 * m ** 3).sum())}
    if call == "train":
        rs = np.random.RandomState(case["elections"])
        N = float(rs.randint(case["m_lo"], case["m_hi"] + 1, case["elections"]).sum())
        return {"bytes": 4 * (17 * N + 7 * 5313), "flops": 6 * 5248 * N}
    m, n, k = float(case["m"]), float(case["n"]), float(min(case["k"], case["m"]))
    if call == "fast":
        return {"bytes": 4 * (m * m + m), "flops": 11 * m * m}
    nw = float(_listed(case))
    pairs = n * m * m if call == "weak" else n * k * k / 2
    byts = {"run": 4 * (n * k + 2 * m * m + 3 * m), "label": 4 * (n * k + 2 * m * m + 19 * m),
            "run_host": 4 * (n * k + 2 * m), "weak": 4 * (n * m + 2 * m * m + 2 * m)}[call]
    return {"bytes": byts, "flops": pairs + 2 * nw ** 3 + (11 * m * m if call == "label" else 0)}


# ------------------------------------------------------------------ in 64 bits

def _tally64(pos):
    n, m = pos.shape
    d = torch.empty((m, m), dtype=torch.int64, device=DEV)
    step = max(1, (1 << 28) // max(1, n * m))
    for i in range(0, m, step):
        d[i:i + step] = (pos[:, i:i + step, None] < pos[:, None, :]).sum(0)
    return d


def _paths64(d, margin):
    p = torch.where(d > d.t(), d - d.t() if margin else d, torch.zeros_like(d))
    for k in range(p.shape[0]):
        torch.maximum(p, torch.minimum(p[:, k:k + 1], p[k:k + 1, :]), out=p)
    return p.fill_diagonal_(0)


def _ranking64(p):
    bb = (p.t() > p).sum(1)
    m = p.shape[0]
    return (bb == 0).long(), torch.argsort(bb * m + torch.arange(m, device=DEV)), bb


def _features64(d, n):
    m = d.shape[0]
    x = d.double()
    off = ~torch.eye(m, dtype=torch.bool, device=DEV)
    diff = x - x.t()
    wo, wi = torch.where(diff > 0, x, 0.0), torch.where(diff < 0, x.t(), 0.0)
    wins, losses = (diff > 0).sum(1).double(), (diff < 0).sum(1).double()
    row, col = x.sum(1), x.sum(0)
    inf = float("inf")
    mo, mi = wo.amax(1), wi.amax(1)
    net = wins - losses

    def ahead(v):
        s = torch.sort(v).values
        return (m - torch.searchsorted(s, v, right=True)).double()

    f = [wins / (m - 1), losses / (m - 1), (m - 1 - wins - losses) / (m - 1), row / (n * (m - 1)), col / (n * (m - 1)),
         mo / n, mi / n, (mi > mo).double(), (mo - mi) / n, wo.sum(1) / (n * (m - 1)), wi.sum(1) / (n * (m - 1)),
         torch.where(off, diff, inf).amin(1) / n, torch.where(off, diff, -inf).amax(1) / n, x.amax(1) / n,
         ahead(row) / (m - 1), ahead(net) / (m - 1)]
    return torch.stack(f, 1)


def _train64(st):
    th = st["theta"].double().requires_grad_()
    x = st["feat"].double()
    h1 = torch.relu(x @ th[0:1024].view(64, 16).t() + th[1024:1088])
    h2 = torch.relu(h1 @ th[1088:5184].view(64, 64).t() + th[5184:5248])
    s = h2 @ th[5248:5312] + th[5312]
    seg = st["seg"].tolist()
    loss = 0.0
    for a, b in zip(seg, seg[1:]):
        t = st["label"][a:b].double()
        loss = loss - (torch.log_softmax(s[a:b], 0) * t / t.sum()).sum()
    loss = loss / (len(seg) - 1)
    g, = torch.autograd.grad(loss, th)
    m1 = 0.9 * st["m1"].double() + 0.1 * g
    m2 = 0.999 * st["m2"].double() + 0.001 * g * g
    mh, vh = m1 / (1 - 0.9 ** st["step"]), m2 / (1 - 0.999 ** st["step"])
    return {"params": st["theta"].double() - st["lr"] * mh / (vh.sqrt() + 1e-8), "adam_m": m1, "adam_v": m2,
            "loss": loss.detach().reshape(1), "grad": g}


def exact(case, seed):
    call = case["call"]
    g = _gen(seed)
    if call == "train":
        return _train64(_train_inputs(case, g))
    if call == "batch" or case["m"] > 4096:
        return None  # counted and closed in 64 bits, these take too long
    ranks = _ballots(case, g)
    d = _tally64(_positions(ranks, case["m"], case.get("tier", 1)))
    p = _paths64(d, bool(case.get("margin")))
    winners, order, bb = _ranking64(p)
    if call == "fast":
        return {"winners": winners, "stats": [None] * 4}
    if call == "run_host":
        return {"winners": winners, "order": order}
    if call == "weak":
        return {"d": d, "p": p, "order": order, "beaten_by": bb}
    out = {"d": d, "p": p, "winners": winners, "order": order, "beaten_by": bb}
    if call == "label":
        out["feat"] = _features64(d, case["n"])
    return out
