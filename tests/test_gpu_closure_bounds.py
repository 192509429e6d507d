"""The persistent closure's tile bounds (skipped updates) and its relabeling
by strength, against the oracle's widths bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_parity import cu, eq, host, lib  # noqa: F401 (the fixture builds the library)

pytestmark = pytest.mark.gpu

NT = 16


def counts(kind, m, top, seed):
    """A count matrix with zero diagonal and entries in [0, top]."""
    rs = np.random.Generator(np.random.PCG64(seed))
    u = np.arange(m)
    if kind == "order":  # close to an order (few edges against it), shuffled
        d = np.where(u[:, None] < u[None, :], top - (u[None, :] - u[:, None]) % max(1, top // 2), 0)
        back = rs.random((m, m)) < 0.001
        d = np.where(back & (u[:, None] > u[None, :]), rs.integers(1, top + 1, (m, m)), d)
        s = rs.permutation(m)
        d = d[np.ix_(s, s)]
    elif kind == "ties":  # few distinct widths, dense: most updates change something
        d = rs.integers(0, 4, (m, m)) * (top // 4)
    elif kind == "chain":  # one heavy cycle through everyone over light random edges
        d = rs.integers(0, max(2, top // 100), (m, m))
        s = rs.permutation(m)
        d[s, np.roll(s, -1)] = top - (u % 7)
    else:  # "sparse": two thirds of the candidates have no edge at all (cold rows and columns)
        d = rs.integers(0, top + 1, (m, m))
        cold = rs.permutation(m)[: 2 * m // 3]
        d[cold, :] = 0
    d = d.astype(np.int32)
    np.fill_diagonal(d, 0)
    return d


@pytest.mark.parametrize("top,flags", [(30000, 0), (30000, 1), (1 << 30, 0)])
@pytest.mark.parametrize("kind,m", [("order", 257), ("order", 1000), ("ties", 320), ("ties", 705), ("chain", 449),
                                    ("chain", 1089), ("sparse", 1200), ("order", 4300)])
def test_closure_tile_bounds(kind, m, top, flags):
    """Squares on both sides of whole tiles, with one tile and with several
    tiles per work item (m = 4300), bounds that need rounding to the progress
    word's 26 bits (2^30), cold rows and columns inside the last warm tile."""
    import paper_2505_12976_gb300 as S
    d = counts(kind, m, top, 7 * m + flags)
    want = oracle.strongest_paths(d, nthreads=NT)
    eq(host(S.schulze_strongest_paths(cu(d), top, flags=flags)), want, f"{kind} m={m} top={top} flags={flags}")
    assert S.context().status() == S.OK


def test_closure_runs_of_neighbouring_tiles():
    """A square in which nearly every update is needed, large enough that a
    work item is a run of neighbouring tiles (two here, the last item of a
    round shorter), in both lane formats, with and without bounds that need
    rounding."""
    import paper_2505_12976_gb300 as S
    m = 3905
    rs = np.random.Generator(np.random.PCG64(m))
    d = rs.integers(0, 30001, (m, m)).astype(np.int32)
    np.fill_diagonal(d, 0)
    want = oracle.strongest_paths(d, nthreads=NT)
    for flags in (0, S.F_FORCE_S32):
        eq(host(S.schulze_strongest_paths(cu(d), 30000, flags=flags)), want, f"flags={flags}")
    big = 1 << 15  # the same order of widths above 2^26
    eq(host(S.schulze_strongest_paths(cu(d * big), 30000 * big)), want * big, "scaled")
    assert S.context().status() == S.OK


def test_run_relabels_listed_candidates_by_ballots():
    """More listed candidates than the cluster closure takes, some unlisted:
    the closure sorts the tally's relabeling by ballots."""
    import paper_2505_12976_gb300 as S
    rs = np.random.Generator(np.random.PCG64(5))
    m, n, k = 900, 4000, 12
    w = np.zeros(m)
    w[rs.permutation(m)[:600]] = (1 + np.arange(600)) ** -0.8
    g = np.where(w > 0, np.log(np.maximum(w, 1e-300)), -1e9)[None, :] + rs.gumbel(size=(n, m))
    r = np.argsort(-g, axis=1)[:, :k].astype(np.int32)
    d, p, win, order, bb = oracle.schulze(r, m)
    out = S.schulze_run(cu(r), m)
    for key, want in (("d", d), ("p", p), ("winners", win), ("order", order), ("beaten_by", bb)):
        eq(host(out[key]), want, key)


def near_top(m, top, seed):
    """Widths of top - 1 between everyone, and of top along a few heavy
    chains over several tiles: what the heavy edges add shows only in the last
    bit below the bound."""
    rs = np.random.Generator(np.random.PCG64(seed))
    u = np.arange(m)
    ahead = (u[None, :] - u[:, None]) % m
    d = np.where((ahead > 0) & (ahead <= (m - 1) // 2), top - 1, 0)  # the next half of the circle: a tournament
    for _ in range(4):
        a = rs.permutation(m)[:9]
        d[a[:-1], a[1:]], d[a[1:], a[:-1]] = top, 0
    np.fill_diagonal(d, 0)
    return d.astype(np.int32)


NEAR_TOP = [(1 << 26) - 1, 1 << 26, (1 << 27) - 1, 1 << 27, (1 << 28) - 3, (1 << 30) - 1, (1 << 31) - 1]


@pytest.mark.parametrize("top", NEAR_TOP)
@pytest.mark.parametrize("m", [257, 513])
def test_closure_bounds_at_the_top_of_the_range(m, top):
    """Entries in the last few values below a power of two, the largest int32
    included: the progress word's rounded maximum must not pass for less."""
    import paper_2505_12976_gb300 as S
    d = near_top(m, top, m)
    got = host(S.schulze_strongest_paths(cu(d), top))
    eq(got, oracle.strongest_paths(d, nthreads=NT), f"m={m} top={top}")
    if m == 257:  # one pair of heavy edges over three tiles
        d = np.triu(np.full((m, m), top - 1, np.int64), 1).astype(np.int32)
        d[0, 70] = d[70, 200] = top
        got = host(S.schulze_strongest_paths(cu(d), top))
        assert got[0, 200] == top
        eq(got, oracle.strongest_paths(d, nthreads=NT), f"three tiles, top={top}")
    assert S.context().status() == S.OK


@pytest.mark.parametrize("top", NEAR_TOP)
def test_beaten_by_at_the_top_of_the_range(top):
    """The closure's own beaten_by, which decides whole tiles by the same
    bounds: the levels of the iterated ranking on widths one apart."""
    import paper_2505_12976_gb300 as S
    d = near_top(300, top, 11)
    want, nlevels = oracle.ranking_iterated(d)
    got, n = S.schulze_ranking_iterated(cu(d), top)
    eq(host(got), want, f"levels, top={top}")
    assert n == nlevels and S.context().status() == S.OK
