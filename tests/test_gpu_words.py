"""The verification kernel's filter on words of nodes, and the three-string test of many nodes at
once, against the oracle: groups of fewer than five positions, one to three groups, full words and
words of one node, rows of one entry, in shared and in global memory, a warp's words in 8, 16 and 32
lanes, n = 1 and 2."""
import numpy as np
import pytest

import planted_inputs as pi
import paper_2403_00306_gb300 as pms

pytestmark = pytest.mark.gpu

# (n, m, l, d)
CASES = [(1, 5, 4, 1), (2, 3, 3, 0), (3, 6, 5, 1), (4, 8, 7, 2), (1, 12, 10, 2), (2, 14, 11, 2), (5, 33, 9, 0),
         (6, 60, 10, 3), (8, 60, 14, 4), (5, 40, 12, 5), (20, 20, 15, 4), (12, 47, 15, 5), (64, 24, 16, 4), (6, 30, 17, 5), (10, 30, 20, 5), (5, 64, 32, 3),
         (2, 19, 19, 6)]


@pytest.mark.parametrize("case", CASES, ids=str)
def test_words_match_oracle(oracle_, case):
    n, m, l, d = case
    for seqs in (pi.planted_instance(n, m, l, d, 3).seqs, pi.random_sequences(n, m, 31)):
        want = oracle_.solve_packed(seqs, l, d)
        for opts in ({}, {"smem_rows": 8}, {"triple_rows": 6}, {"triple_rows": -1}, {"chunk_work": 4096}):
            with pms.Context(0) as c:
                c.set_options(grab=1, **opts)
                assert np.array_equal(c.solve(seqs, l, d), want), opts


@pytest.mark.parametrize("case", [(20, 900, 15, 4), (20, 600, 17, 5), (12, 260, 19, 6), (20, 200, 13, 4), (20, 600, 14, 4)], ids=str)
def test_words_and_batches_agree(case):
    """Whole motif sets of larger instances: words of nodes ((14,4): the walk) against breadth-first batches."""
    n, m, l, d = case
    seqs = pi.planted_instance(n, m, l, d, 9).seqs
    got = []
    for opts in ({"grab": 1}, {"grab": 128}, {"grab": 1, "triple_rows": 19}):
        with pms.Context(0) as c:
            c.set_options(**opts)
            got.append(c.solve(seqs, l, d))
    assert len(got[0]) > 0
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])


def test_walk_and_words_in_one_launch(oracle_):
    """Batches in tree form of instances with words of nodes ((15,4), (17,5)), of instances whose nodes are
    walked one by one ((9,2), (13,4), (12,3)) and of both."""
    words = [(pi.planted_instance(8, 60, 15, 4, 3).seqs, 15, 4), (pi.planted_instance(6, 30, 17, 5, 4).seqs, 17, 5)]
    walk = [(pi.planted_instance(5, 400, 9, 2, 5).seqs, 9, 2), (pi.planted_instance(10, 220, 13, 4, 6).seqs, 13, 4),
            (pi.planted_instance(6, 500, 12, 3, 7).seqs, 12, 3)]
    with pms.Context(0) as c:
        c.set_options(grab=1)
        for batch in (words, walk, [walk[0], words[0], walk[1], words[1], walk[2], words[0]]):
            for (seqs, l, d), got in zip(batch, c.solve_batch(batch)):
                assert np.array_equal(got, oracle_.solve_packed(seqs, l, d)), (l, d)


def test_memory_budget_that_holds_the_walk(oracle_):
    """A budget that the batches of nodes just fit also does for the default filter: its table of words,
    24 KB here, is left out then."""
    seqs = pi.planted_instance(6, 26, 19, 6, 4).seqs
    want = oracle_.solve_packed(seqs, 19, 6)

    def fits(budget, **opts):
        with pms.Context(0, mem_budget_bytes=budget) as c:
            c.set_options(max_motifs=1 << 12, **opts)
            try:
                return c.solve(seqs, 19, 6)
            except pms.PMSError as e:
                assert e.code == pms.PMS_ENOMEM
    lo, hi = 1 << 12, 1 << 24
    assert fits(lo, grab=32) is None and fits(hi, grab=32) is not None
    while hi - lo > 256:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(mid, grab=32) is not None else (mid, hi)
    for opts in ({"grab": 32}, {"grab": 1}):
        got = fits(hi, **opts)
        assert got is not None and np.array_equal(got, want), opts


@pytest.mark.parametrize("case", [(5, 144, 14, 4), (4, 60, 12, 3), (6, 90, 15, 3), (12, 200, 10, 2), (8, 150, 13, 1)], ids=str)
def test_repetitive_sequences_match_oracle(oracle_, case):
    """Runs of one letter and repeats of seven: seeds that occur in every sequence, all of whose nodes pass."""
    n, m, l, d = case
    runs = pi.planted_instance(n, m, l, d, 23).seqs.copy()
    runs[:, m // 4:m // 2] = ord("A")
    repeats = pi.random_sequences(n, m, 24).copy()
    repeats[:, m // 3:2 * m // 3] = np.resize(np.frombuffer(b"GATTACA", dtype=np.uint8), 2 * m // 3 - m // 3)
    for seqs in (runs, repeats):
        want = oracle_.solve_packed(seqs, l, d)
        with pms.Context(0) as c:
            c.set_options(grab=1)
            assert np.array_equal(c.solve(seqs, l, d), want)
            assert np.array_equal(c.solve_batch([(seqs, l, d)] * 2)[1], want)
