"""The position-compare tally on bit planes against the oracle: edges of the
64 x 64 tiles, of 32-ballot groups, of the 2048-candidate turns and of the
position widths."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from test_gpu_parity import cu, eq, host, lib  # noqa: F401 (the fixture builds the library)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 200])
@pytest.mark.parametrize("m", [1, 2, 63, 64, 65, 128, 129, 257])
def test_dense_tally_tiles_and_groups(m, n):
    import paper_2505_12976_gb300 as S
    full = W.impartial(m * 1000 + n, n, m)
    eq(host(S.schulze_tally(cu(full), m, flags=S.F_TALLY_DENSE)), oracle.tally(full, m), "full")
    for k in {max(1, m - 1), max(1, m // 2)}:  # one or many unlisted candidates, at position k
        part = np.ascontiguousarray(full[:, :k])
        eq(host(S.schulze_tally(cu(part), m, flags=S.F_TALLY_DENSE)), oracle.tally(part, m), f"top-{k}")


@pytest.mark.parametrize("m", [2047, 2048, 2113])
def test_dense_tally_candidate_turns(m):
    import paper_2505_12976_gb300 as S
    full = W.impartial(m, 70, m)
    eq(host(S.schulze_tally(cu(full), m)), oracle.tally(full, m), "full")
    bad = full.copy()
    bad[41, m - 1] = bad[41, 3]  # a repeated id, in whichever turn holds it
    S.schulze_tally(cu(bad), m)
    assert S.context().status() == S.EDATA
    bad[41, m - 1] = m
    S.schulze_tally(cu(bad), m)
    assert S.context().status() == S.EDATA


@pytest.mark.parametrize("top", [0, 1, 2, 255, 256, 32767, 32768, 65534])
def test_positions_of_every_width(top):
    """Largest positions on both sides of a bit, and more than one chunk of
    ballots' worth of splits."""
    import paper_2505_12976_gb300 as S
    rs = np.random.Generator(np.random.PCG64(top + 1))
    pos = rs.integers(0, top + 1, (333, 70)).astype(np.int32)
    pos[17, 5] = top
    eq(host(S.schulze_tally_positions(cu(pos))), oracle.tally_positions(pos), f"top={top}")
    for wrong in (-1, 65535):
        pos[200, 69] = wrong
        S.schulze_tally_positions(cu(pos))
        assert S.context().status() == S.EDATA


def test_dense_tally_several_chunks():
    """More ballots than one chunk of planes (65536)."""
    import paper_2505_12976_gb300 as S
    full = W.impartial(9, 65536 + 37, 9)
    eq(host(S.schulze_tally(cu(full), 9)), oracle.tally(full, 9), "two chunks")
