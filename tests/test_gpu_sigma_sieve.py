"""The general-alphabet search with d <= 4 and q = n (tuples of a node's letters in a bit map) against
the oracle, at its edges: nodes of 0 to 4 letters, alphabets of 3 to 32, maps of one and two sizes,
rows whose masks share a word with their letters or not, more rows than a list, a sequence or shared
memory holds, more row masks than are kept."""
import numpy as np
import pytest

import planted_inputs as pi
import paper_2403_00306_gb300 as pms

pytestmark = pytest.mark.gpu

ALPHABET = b"ACDEFGHIKLMNPQRSTVWYBJOUXZabcdef"

# (sigma, l, d, n, m)
CASES = [(3, 6, 4, 9, 40), (3, 16, 4, 6, 60), (4, 5, 4, 3, 20), (4, 8, 3, 12, 70), (5, 7, 4, 10, 33), (8, 6, 4, 8, 50),
         (20, 5, 4, 20, 7), (20, 6, 4, 6, 18), (20, 9, 0, 3, 40), (20, 7, 1, 4, 50), (20, 8, 2, 5, 60), (20, 9, 3, 6, 50),
         (20, 12, 3, 4, 60), (22, 5, 3, 5, 24), (23, 5, 3, 5, 24), (32, 5, 3, 4, 20), (32, 5, 4, 10, 6), (32, 12, 2, 3, 40),
         (4, 5, 3, 64, 60), (4, 32, 4, 3, 40), (4, 6, 4, 6, 450), (20, 9, 1, 64, 1100), (20, 4, 3, 3, 9)]


@pytest.mark.parametrize("case", CASES, ids=str)
def test_matches_oracle(oracle_, case):
    sigma, l, d, n, m = case
    alphabet = ALPHABET[:sigma]
    inst = pi.planted_instance_sigma(n, m, l, min(d, l), 5, alphabet)
    want = oracle_.sigma_solve(inst.seqs, l, d, alphabet)
    with pms.Context(0) as c:
        got = c.solve_sigma(inst.seqs, l, d, alphabet)
        assert np.array_equal(got, want), (len(got), len(want))
        c.set_options(ctas_per_sm=1, smem_rows=8)    # few CTAs, rows in global scratch
        assert np.array_equal(c.solve_sigma(inst.seqs, l, d, alphabet), want)


# few sequences, whose windows several warps share (W around multiples of 128 and of their shares), and answers
# of many strings a node
FEW = [(20, 4, 2, 2, 140), (20, 5, 3, 2, 14), (4, 7, 4, 2, 300), (4, 6, 2, 3, 270), (3, 8, 3, 5, 135), (32, 4, 2, 2, 50),
       (23, 5, 2, 2, 70), (20, 6, 1, 4, 700), (4, 9, 2, 2, 1300), (20, 6, 2, 9, 260), (20, 9, 1, 2, 2100), (4, 8, 3, 4, 519),
       (20, 7, 4, 2, 9), (4, 6, 4, 8, 133), (5, 6, 0, 2, 1029), (20, 6, 3, 3, 8)]


@pytest.mark.parametrize("case", FEW, ids=str)
def test_few_sequences_and_dense_answers_match_oracle(oracle_, case):
    sigma, l, d, n, m = case
    alphabet = ALPHABET[:sigma]
    inst = pi.planted_instance_sigma(n, m, l, d, 6, alphabet)
    want = oracle_.sigma_solve(inst.seqs, l, d, alphabet)
    with pms.Context(0) as c:
        c.set_options(max_motifs=1 << 22)
        assert np.array_equal(c.solve_sigma(inst.seqs, l, d, alphabet), want)
        c.set_options(max_motifs=1 << 22, ctas_per_sm=1, smem_rows=8)
        assert np.array_equal(c.solve_sigma(inst.seqs, l, d, alphabet), want)


def test_memory_budget_that_holds_the_depth_first_form():
    """A budget that a quorum of n - 1 (searched depth first) just fits also does for q = n: its own buffers
    (packed letters, and rows in global memory, more than fit on chip here) are not asked for then."""
    seqs = pi.planted_instance_sigma(3, 500, 9, 2, 4).seqs
    with pms.Context(0) as c:
        want = c.solve_sigma(seqs, 9, 2)
    def fits(budget, q):
        with pms.Context(0, mem_budget_bytes=budget) as c:
            try:
                got = c.solve_sigma(seqs, 9, 2, q=q)
            except pms.PMSError as e:
                assert e.code == pms.PMS_ENOMEM
                return None
            return got
    lo, hi = 1 << 20, 1 << 26
    assert fits(lo, 2) is None and fits(hi, 2) is not None
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(mid, 2) is not None else (mid, hi)
    got = fits(hi, 0)
    assert got is not None and np.array_equal(got, want)
