"""Edges of the kernels that a dispatch picks by size: the small closure (one
cluster launch), the blocks of the propagation, the batch's bit planes, the
training step's split reduction and the host call's graph."""
import numpy as np
import pytest
import torch

import oracle
import oracle.mlp as M
import workloads as W
from test_gpu_closure_bounds import counts
from test_gpu_parity import cu, eq, host, lib  # noqa: F401 (the fixture builds the library)

pytestmark = pytest.mark.gpu


def shifted(a):
    """The same matrix on the device, 4 bytes off a 16-byte boundary."""
    buf = torch.zeros(a.size + 1, dtype=torch.int32, device="cuda")
    buf[1:] = cu(a).reshape(-1)
    return buf[1:].view(a.shape)


# ------------------------------------------------- closure of few candidates

@pytest.mark.parametrize("m", [1, 2, 7, 8, 9, 63, 64, 65, 127, 191, 192, 193, 255, 256, 257])
def test_small_closure_both_lanes_margin_and_alignment(m):
    """Sizes around its blocks and around both of its limits (192 with 32-bit
    lanes, 256 with 16-bit ones), against the oracle; the last sizes take the
    general path, which has to agree."""
    import paper_2505_12976_gb300 as S
    d = counts("ties", m, 30000, m) if m > 2 else np.array([[0, 5], [3, 0]], np.int32)[:m, :m]
    for margin in (0, S.F_MARGIN):
        w = oracle.weights_margin(d) if margin else oracle.weights(d)
        want = oracle.closure(w, nthreads=4)
        for lanes in (1, 2):
            what = f"m={m} margin={margin} lanes={lanes}"
            eq(host(S.schulze_strongest_paths(cu(d), 30000, flags=lanes | margin)), want, what)
            eq(host(S.schulze_strongest_paths(shifted(d), 30000, flags=lanes | margin, p=shifted(0 * d))), want,
               what + " unaligned")
            eq(host(S.schulze_strongest_paths_static(cu(d), 30000, flags=lanes | margin)), want, what + " static")
    assert S.context().status() == S.OK


@pytest.mark.parametrize("m", [1, 2, 3, 31, 64, 65, 128, 129, 130, 191, 192, 255, 256])
def test_small_closure_with_few_candidates_with_edges(m):
    """No candidate with an edge, one, a few, two neighbours, the last ones,
    about half, all but one, and on both sides of the line at which the square
    is filled anew."""
    import paper_2505_12976_gb300 as S
    rs = np.random.Generator(np.random.PCG64(m))
    full = counts("ties", m, 30000, m) if m > 2 else np.array([[0, 5], [3, 0]], np.int32)[:m, :m]
    sets = [[], [0], [m - 1], [m - 2, m - 1], rs.permutation(m)[:5], rs.permutation(m)[:m // 4], rs.permutation(m)[:m // 2],
            np.arange(0, m, 2), np.arange(1, m, 2), rs.permutation(m)[:max(0, m - 1)]]
    line = -(-2400 // m)  # candidates without an edge
    sets += [rs.permutation(m)[:max(0, m - line + x)] for x in (0, 1)]
    for t, keep in enumerate(sets):
        d = np.zeros_like(full)
        keep = np.unique(np.clip(np.array(keep, np.int64), 0, m - 1))
        d[keep] = full[keep] + rs.integers(0, 50, (len(keep), m))
        np.fill_diagonal(d, 0)
        for flags in (0, 1, S.F_MARGIN):
            w = oracle.weights_margin(d) if flags == S.F_MARGIN else oracle.weights(d)
            want = oracle.closure(w, nthreads=2)
            eq(host(S.schulze_strongest_paths(cu(d), 30100, flags=flags)), want, f"m={m} set {t} flags={flags}")
    assert S.context().status() == S.OK


@pytest.mark.parametrize("m,n,k", [(1, 4, 1), (2, 5, 1), (8, 30, 8), (65, 50, 64), (192, 40, 192), (193, 60, 20),
                                   (256, 90, 256), (257, 90, 256)])
@pytest.mark.parametrize("flags", [0, 1, 32])
def test_small_run_winners_and_ranking(m, n, k, flags):
    import paper_2505_12976_gb300 as S
    r = W.impartial(m + 3 * n, n, m, k)
    d = oracle.tally(r, m)
    p = oracle.closure(oracle.weights_margin(d) if flags & 32 else oracle.weights(d), nthreads=4)
    order, bb = oracle.ranking(p)
    out = S.schulze_run(cu(r), m, flags=flags)
    for key, want in (("d", d), ("p", p), ("winners", oracle.winners(p)), ("order", order), ("beaten_by", bb)):
        eq(host(out[key]), want, f"{key} m={m} flags={flags}")


@pytest.mark.parametrize("m", [2, 64, 150])
@pytest.mark.parametrize("wrong", [-1, 101])
def test_small_closure_reports_counts_out_of_range(m, wrong):
    import paper_2505_12976_gb300 as S
    d = np.minimum(counts("ties", m, 100, 3), 100) if m > 2 else np.array([[0, 5], [3, 0]], np.int32)
    d[m - 1, 0] = wrong
    S.schulze_strongest_paths(cu(d), 100)
    assert S.context().status() == S.EDATA
    S.schulze_strongest_paths(cu(np.abs(d) % 101), 100)
    assert S.context().status() == S.OK


@pytest.mark.parametrize("m", [257, 300, 705])
@pytest.mark.parametrize("bound,wrong", [(100, -1), (100, 101), (100, -2**31), (40000, 40001), (2**31 - 1, -1),
                                         (2**40, -5), (0, 1)])
def test_large_closure_reports_counts_out_of_range(m, bound, wrong):
    """One entry below 0 or above the bound is reported, wherever it lies and
    whatever the bound (beyond 31 bits too); the largest allowed one is not."""
    import paper_2505_12976_gb300 as S
    ok = min(bound, 2**31 - 1)
    d = np.minimum(counts("ties", m, 100, 3), ok).astype(np.int32)
    for i, j in ((0, m - 1), (m - 1, 0), (m // 2, m // 2 + 1), (m - 1, m - 1)):
        for flags in (0, S.F_MARGIN):
            e = d.copy()
            e[i, j] = wrong
            S.schulze_strongest_paths(cu(e), bound, flags=flags)
            assert S.context().status() == S.EDATA, (i, j, flags)
            e[i, j] = ok
            S.schulze_strongest_paths(shifted(e), bound, flags=flags)
            assert S.context().status() == S.OK, (i, j, flags)


@pytest.mark.parametrize("m,odd", [(701, 0), (704, 1), (1000, 0)])
def test_general_path_beaten_by_with_cold_columns(m, odd):
    """winners, order and beaten_by of the general path with candidates that
    have no edge, odd rows or an unaligned base."""
    import paper_2505_12976_gb300 as S
    d = counts("sparse", m, 900, m + odd)
    p = oracle.strongest_paths(d, nthreads=16)
    order, bb = oracle.ranking(p)
    dd = shifted(d) if odd else cu(d)
    pg = S.schulze_strongest_paths(dd, 900)
    eq(host(pg), p, "p")
    got = S.schulze_ranking(shifted(p) if odd else pg)
    eq(host(got[0]), order, "order")
    eq(host(got[1]), bb, "beaten_by")
    eq(host(S.schulze_winners(pg)), oracle.winners(p), "winners")


@pytest.mark.parametrize("listed,unlisted", [(300, 0), (257, 63), (257, 64), (320, 1), (321, 127), (321, 200),
                                             (449, 300), (2113, 70)])
@pytest.mark.parametrize("lanes", [1, 2])
def test_run_beaten_by_of_large_squares_without_hint(listed, unlisted, lanes):
    """beaten_by as the closure counts it from its tiles and their bounds: a
    dense tally of short lists gives no hint, so the unlisted candidates are
    general cold columns, inside the last warm tile, beyond it, or both;
    popular and unpopular candidates far apart, so that whole tiles beat whole
    tiles; more than 32 tile rows at the last size."""
    import paper_2505_12976_gb300 as S
    m, n, k = listed + unlisted, min(40 * listed, 30000), 6
    rs = np.random.Generator(np.random.PCG64(7 * listed + unlisted))
    ids = rs.permutation(m)[:listed]
    # ballots around an order of the listed candidates: windows of neighbours, popular ones first
    start = np.minimum((listed - k) * rs.random(n) ** 1.5, listed - k).astype(np.int64)
    start[: listed - k + 1] = np.arange(listed - k + 1)  # everyone is on a ballot
    r = ids[start[:, None] + np.argsort(np.arange(k)[None, :] + rs.gumbel(size=(n, k)), axis=1)].astype(np.int32)
    d, p, win, order, bb = oracle.schulze(r, m, nthreads=16)
    out = S.schulze_run(cu(r), m, flags=S.F_TALLY_DENSE | lanes)
    for key, want in (("d", d), ("p", p), ("beaten_by", bb), ("order", order), ("winners", win)):
        eq(host(out[key]), want, f"{key} listed={listed} unlisted={unlisted} lanes={lanes}")
    assert S.context().status() == S.OK


@pytest.mark.parametrize("m", [4096, 5376, 5377, 6400])
def test_run_ranking_on_both_sides_of_its_launch_rule(m):
    """order, winners and beaten_by against p on the host, with the counting
    launched early (m up to 5376 on 152 SMs) and plainly, twice in a row on
    other ballots."""
    import paper_2505_12976_gb300 as S
    for seed in (1, 2):
        out = S.schulze_run(cu(W.mallows(seed, 500, m, 20, phi=0.9)), m)
        p = host(out["p"])
        bb = (p.T > p).sum(1).astype(np.int32)
        eq(host(out["beaten_by"]), bb, f"beaten_by m={m}")
        eq(host(out["order"]), np.lexsort((np.arange(m), bb)).astype(np.int32), f"order m={m}")
        eq(host(out["winners"]), (bb == 0).astype(np.int32), f"winners m={m}")


# ------------------------------------------------------ blocks of propagation

@pytest.mark.parametrize("m", [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 200])
@pytest.mark.parametrize("top", [3, 1 << 22])
def test_propagation_block_edges(m, top):
    """Ties everywhere (top = 3) and counts past 16 bits, both weights, with
    rows on and off 16-byte boundaries: winners and rounds as the oracle's."""
    import paper_2505_12976_gb300 as S
    rs = np.random.Generator(np.random.PCG64(m + top))
    d = rs.integers(0, top + 1, (m, m)).astype(np.int32)
    np.fill_diagonal(d, 0)
    for margin in (0, S.F_MARGIN):
        w = oracle.weights_margin(d) if margin else oracle.weights(d)
        win, it, rounds = oracle.winners_pregel(w)
        for dev in (cu(d), shifted(d)):
            got, stats = S.schulze_winners_propagation(dev, flags=margin)
            eq(host(got), win, f"winners m={m} margin={margin}")
            assert stats == [it, rounds], (m, margin)


@pytest.mark.parametrize("m", [257, 500, 1023, 1024, 1025, 1087, 1088, 1089, 1151])
@pytest.mark.parametrize("top", [2000, 1 << 22])
def test_propagation_rows_and_blocks(m, top):
    """The same around the size from which the passes take pairs of blocks
    instead of rows (m = 1025), at edges of the blocks."""
    test_propagation_block_edges(m, top)


# ------------------------------------------------------------ batch bit planes

@pytest.mark.parametrize("per_tile", [1, 2, 4])
def test_batch_plane_groups_and_parts(per_tile):
    """Ballot counts around a group of 32, elections past the planes kept at
    once (8192 ballots), and ballots that list all, all but one or few."""
    import paper_2505_12976_gb300 as S
    els = []
    for t, (n, m) in enumerate([(1, 65), (31, 64), (32, 63), (33, 129), (64, 33), (65, 16), (95, 17), (255, 300),
                                (8191, 40), (8192, 41), (8193, 70), (16390, 9)]):
        for k in sorted({m, m - 1, max(1, m // 4)}):
            els.append((W.impartial(500 + 7 * t + k, n, m, k), m))
    n, m, k = (np.array(x, np.int32) for x in ([r.shape[0] for r, _ in els], [m for _, m in els],
                                               [r.shape[1] for r, _ in els]))
    b = S.SchulzeBatch(n, m, k)
    for bucket in range(5):
        b.set_bucket_tiles(bucket, per_tile)
    out = [torch.full((size,), -3, dtype=torch.int32, device="cuda")
           for size in (b.mat_elems, b.mat_elems, b.vec_elems, b.vec_elems, b.vec_elems)]
    b.run(cu(np.concatenate([r.reshape(-1) for r, _ in els])), *out)
    got = [host(t) for t in out]
    for e, (r, me) in enumerate(els):
        mo, vo = int(b.mat_off[e]), int(b.vec_off[e])
        want = oracle.schulze(r, me)
        for name, g, w, off in zip(("d", "p", "winners", "order", "beaten_by"), got, want, (mo, mo, vo, vo, vo)):
            eq(g[off:off + w.size].reshape(w.shape), w, f"{name} of election {e}: n={len(r)} m={me} k={r.shape[1]}")


@pytest.mark.parametrize("n,v", [(33, 32), (64, 63), (100, 99), (100, 0), (8193, 8192)])
@pytest.mark.parametrize("k", [40, 39, 11])
@pytest.mark.parametrize("fault", ["repeat", "high", "low"])
def test_batch_planes_report_bad_ballots(n, v, k, fault):
    """One wrong id, also in the last ballot of a partial group or of a second
    turn, is reported; the same elections without it are not."""
    import paper_2505_12976_gb300 as S
    m = 40
    r = W.impartial(n + k, n, m, k)
    b = S.SchulzeBatch([n], [m], [k])
    vec = [torch.empty(m, dtype=torch.int32, device="cuda") for _ in range(3)]
    b.run(cu(r), None, None, *vec)
    assert S.context().status() == S.OK
    r[v, k - 1] = {"repeat": r[v, 0], "high": m, "low": -1}[fault]
    b.run(cu(r), None, None, *vec)
    assert S.context().status() == S.EDATA


# ------------------------------------------------------------- training step

@pytest.mark.parametrize("N", [2, 63, 64, 65, 1023, 1024, 1025, 2177])
def test_train_step_chunk_and_segment_edges(N):
    """Candidates around the 64 of a gradient block and around the 16 runs
    that the reduction splits its chunks into; the tolerances are those of
    the step's other test (FP32 sums against float64)."""
    import paper_2505_12976_gb300 as S
    rs = np.random.Generator(np.random.PCG64(N))
    X = rs.random((N, M.NFEAT)).astype(np.float32)
    cuts = np.unique(np.concatenate([[0], rs.integers(1, N, 5) if N > 60 else [], [N]])).astype(np.int32)
    lab = np.zeros(N, np.int32)
    for a, b in zip(cuts[:-1], cuts[1:]):
        lab[rs.integers(a, b)] = 1
    theta = W.mlp_init(5)
    want_loss, want_g, _ = M.loss_and_grad(theta.astype(np.float64), X.astype(np.float64), lab, cuts)
    p = torch.from_numpy(theta.copy()).cuda()
    m1, m2 = (torch.zeros(M.NPARAM, device="cuda") for _ in range(2))
    loss, g = S.schulze_mlp_train_step(p, m1, m2, 1, torch.from_numpy(X).cuda(), cu(lab), cu(cuts), 1e-2)
    scale = np.abs(want_g).max()
    assert loss.item() == pytest.approx(want_loss, rel=1e-5)
    np.testing.assert_allclose(g.cpu().numpy(), want_g, rtol=1e-4, atol=1e-4 * scale)


# ---------------------------------------------------------- host call's graph

@pytest.mark.parametrize("m,n,k", [(30, 200, 30), (700, 900, 12)])
def test_host_call_replays_on_any_buffers(m, n, k):
    """Calls of one size with page-locked, pageable and other buffers in turn,
    each with its own ballots: every call answers for the ballots it got."""
    import paper_2505_12976_gb300 as S
    for t in range(6):
        r = W.impartial(40 + t, n, m, k)
        _, p, win, order, _ = oracle.schulze(r, m, 8)
        src = torch.from_numpy(r.copy())
        if t % 2:
            src = src.pin_memory()
        outs = [torch.full((m,), -9, dtype=torch.int32) for _ in range(2)]
        if t % 3 == 0:
            outs = [x.pin_memory() for x in outs]
        S.schulze_run_host(src, m, winners=outs[0], order=outs[1])
        eq(outs[0].numpy(), win, f"winners, call {t}")
        eq(outs[1].numpy(), order, f"order, call {t}")
    bad = r.copy()
    bad[n - 1, 0] = m
    with pytest.raises(S.SchulzeError):
        S.schulze_run_host(bad, m)
    got, _ = S.schulze_run_host(r, m)
    eq(got, win, "after a refused call")


def test_host_call_captures_a_size_that_comes_back():
    """A graph is made at the second call in a row of one size, never for
    sizes that take turns; the one at hand serves its size in between. Every
    call answers for its own ballots."""
    import paper_2505_12976_gb300 as S
    ctx, m, k = S.context(), 391, 30
    ballots = {n: W.impartial(n, n, m, k) for n in (901, 902, 903)}
    want = {n: oracle.schulze(r, m, 8) for n, r in ballots.items()}

    def call(n, flags=0):
        before = ctx.graph_captures()
        win, order = S.schulze_run_host(ballots[n], m, flags=flags)
        eq(win, want[n][2], f"winners n={n}")
        eq(order, want[n][3], f"order n={n}")
        return ctx.graph_captures() - before

    call(903, flags=1), call(903, flags=1)  # workspace grown, another graph at hand
    got = [call(n) for n in (901, 902, 901, 902, 903, 903, 901, 903, 902, 902, 902)]
    assert got == [0, 0, 0, 0, 0, 1, 0, 0, 0, 1, 0]


@pytest.mark.parametrize("pinned", [False, True])
def test_host_call_counts_and_times_its_launches(pinned):
    """Launch counts and kernel times of the host call do not depend on
    whether a graph serves it."""
    import paper_2505_12976_gb300 as S
    ctx, m, n, k = S.context(), 333, 800, 25
    src = torch.from_numpy(W.impartial(5, n, m, k).copy())
    if pinned:
        src = src.pin_memory()
    counts = []
    for _ in range(4):
        before = ctx.launch_count()
        S.schulze_run_host(src, m)
        counts.append(ctx.launch_count() - before)
    assert counts[0] > 0 and counts == [counts[0]] * 4
    ctx.profile(True)
    for _ in range(3):
        S.schulze_run_host(src, m)
    seen = ctx.profile_read()
    ctx.profile(False)
    assert sum(v["launches"] for v in seen.values()) == 3 * counts[0], seen
    assert seen["closure_persistent"]["launches"] == 3 and seen["closure_persistent"]["ms"] > 0


# ------------------------------------ winners when the warm set is too large

@pytest.mark.parametrize("m,warm,answer", [(2049, 2048, (0, 1)), (2049, 2049, (2,)), (6001, 2048, (0, 1)),
                                           (6001, 2049, (2,)), (6000, 6000, (2,)), (9001, 9001, (2,))])
def test_winners_fast_around_the_warm_limit(m, warm, answer):
    """Candidates with an outgoing edge around the certification's 2048, few
    and many to either side: the features pass may stop once it has seen too
    many, and the propagation then decides, as it does by itself."""
    import paper_2505_12976_gb300 as S
    rs = np.random.Generator(np.random.PCG64(m + warm))
    s = rs.permutation(m)[:warm]  # the warm ones: near an order, and a cycle at the top
    d = np.zeros((m, m), np.int32)
    back = rs.random((warm, warm)) < 1e-4
    base = np.where(np.arange(warm)[:, None] < np.arange(warm)[None, :], rs.integers(600, 900, (warm, warm)), 100)
    d[np.ix_(s, s)] = np.where(back, 950, base)
    d[s[0], s[1]], d[s[1], s[2]], d[s[2], s[0]] = 700, 700, 700
    d[s[1], s[0]] = d[s[2], s[1]] = d[s[0], s[2]] = 100
    if warm < m:
        d[s, [c for c in range(m) if c not in set(s.tolist())][0]] = 500  # the last one has an edge too
    else:
        d[s[-1], s[0]], d[s[0], s[-1]] = 400, 300
    np.fill_diagonal(d, 0)
    dev = cu(d)
    assert int(((dev > dev.T).sum(1) > 0).sum()) == warm
    for params in (None, torch.from_numpy(W.mlp_init(5)).cuda()):
        got, stats = S.schulze_winners_fast(dev, 1000, params)
        assert stats[1] in answer, stats
        eq(host(got), host(S.schulze_winners(S.schulze_strongest_paths(dev, 1000))), f"m={m} warm={warm}")
