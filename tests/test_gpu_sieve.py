"""The sieve form against the oracle, bit-exact, at the edges of its blocks, words and windows,
and against the tree form (which an explicit node filter selects) on larger instances."""
import numpy as np
import pytest

import planted_inputs as pi
import paper_2403_00306_gb300 as pms

pytestmark = pytest.mark.gpu

# l = 8..10: 3 middle letters (8 and 9: almost no prefix); 11: 4; 12, 13: 5, a CTA per block;
# 14 and more: 5, a warp per block, or 6, a CTA per block; W around 32 and one window per sequence;
# more sequences than a CTA has warps; more changes than middle letters
SMALL = [(2, 9, 9, 2), (2, 40, 8, 1), (3, 39, 8, 1), (9, 40, 9, 2), (17, 41, 9, 1), (5, 64, 10, 3), (64, 42, 10, 4),
         (8, 43, 11, 3), (6, 11, 11, 5), (9, 75, 12, 4), (20, 96, 13, 4), (12, 45, 13, 6), (7, 46, 14, 5),
         (10, 60, 15, 5), (5, 16, 16, 4), (12, 50, 16, 6), (4, 300, 14, 4), (10, 290, 15, 5), (20, 80, 16, 6)]
# 5 counter planes up to 31 sequences and l >= 12, else 7
QUORUM = [(5, 60, 9, 1, 3), (12, 64, 10, 2, 10), (31, 50, 12, 3, 28), (32, 50, 12, 3, 29), (64, 40, 11, 3, 60),
          (8, 50, 13, 4, 7), (6, 40, 15, 4, 5), (31, 300, 13, 4, 29), (10, 48, 16, 5, 9), (4, 30, 9, 2, 1)]


@pytest.mark.parametrize("case", SMALL, ids=str)
def test_sieve_matches_oracle(oracle_, case):
    n, m, l, d = case
    for seqs in (pi.planted_instance(n, m, l, d, 7).seqs, pi.random_sequences(n, m, 70)):
        want = oracle_.solve_packed(seqs, l, d)
        with pms.Context(0) as c:
            assert np.array_equal(c.solve(seqs, l, d), want)
            for got in c.solve_batch([(seqs, l, d)] * 3):   # a warp per block for every l
                assert np.array_equal(got, want)


@pytest.mark.parametrize("case", QUORUM, ids=str)
def test_sieve_quorum_matches_oracle(oracle_, case):
    n, m, l, d, q = case
    seqs = pi.planted_instance(n, m, l, d, 11).seqs
    with pms.Context(0) as c:
        c.set_options(quorum=q)
        assert np.array_equal(c.solve(seqs, l, d), oracle_.solve_quorum(seqs, l, d, q, cap=1 << 24))


@pytest.mark.parametrize("case", [(9, 2, 20, 600, 0), (11, 3, 17, 733, 0), (12, 3, 25, 1000, 0), (13, 4, 20, 600, 0),
                                  (14, 4, 13, 999, 0), (15, 4, 20, 1100, 0), (15, 5, 20, 301, 0), (16, 5, 20, 250, 0),
                                  (17, 5, 20, 1150, 0), (18, 6, 20, 400, 0),
                                  (13, 4, 20, 300, 18), (15, 4, 15, 200, 12), (12, 3, 40, 400, 37)], ids=str)
def test_sieve_and_tree_form_agree(case):
    """Whole motif sets and, on the device entry point, raw counts (a motif once per seed window near it)."""
    import torch
    l, d, n, m, q = case
    seqs = pi.planted_instance(n, m, l, d, 3).seqs
    d_in = torch.from_numpy(seqs.copy()).cuda()
    outs = []
    for opts in ({}, {"grab": 1}):
        with pms.Context(0) as c:
            c.set_options(quorum=q, **opts)
            out = torch.zeros(1 << 16, dtype=torch.int64, device="cuda")
            st = torch.zeros(4, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            for _ in range(3):   # kernel by kernel, captured, replayed
                c.solve_device(d_in, n, m, l, d, out, 1 << 16, st)
            torch.cuda.synchronize()
            outs.append((out.cpu().numpy(), st.cpu().numpy(), c.solve(seqs, l, d)))
    assert np.array_equal(outs[0][1], outs[1][1]) and np.array_equal(outs[0][0], outs[1][0])
    assert np.array_equal(outs[0][2], outs[1][2]) and len(outs[0][2]) > 0


@pytest.mark.parametrize("case", [(9, 2, 12, 900, 0), (10, 3, 20, 500, 0), (11, 3, 12, 700, 0), (13, 4, 16, 900, 0),
                                  (14, 4, 6, 900, 0), (11, 3, 14, 600, 13)], ids=str)
def test_large_answers_sorted_by_buckets(case):
    """Answers of a thousand to a few hundred thousand motifs (motifs of fewer and of more letters than
    a bucket number holds), alone, in a batch and on the device entry point with too little room."""
    import torch
    l, d, n, m, q = case
    seqs = pi.planted_instance(n, m, l, d, 21).seqs
    with pms.Context(0) as c, pms.Context(0) as tree:
        c.set_options(quorum=q)
        tree.set_options(quorum=q, grab=1)
        want = tree.solve(seqs, l, d)
        assert len(want) > 1000
        assert np.array_equal(c.solve(seqs, l, d), want)
        for got in c.solve_batch([(seqs, l, d)] * 3):
            assert np.array_equal(got, want)
        out = torch.zeros(1024, dtype=torch.int64, device="cuda")
        st = torch.zeros(4, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        c.solve_device(torch.from_numpy(seqs.copy()).cuda(), n, m, l, d, out, 1000, st)
        torch.cuda.synchronize()
        s = st.cpu().numpy().astype(np.uint32)
        assert s[1] == len(want) and s[2] == 2
        assert np.array_equal(out[:1000].cpu().numpy().astype(np.uint64), want[:1000]) and not out[1000:].any()


@pytest.mark.parametrize("case", [(45, 300, 9, 1), (64, 120, 10, 2), (50, 500, 11, 2)], ids=str)
def test_blocks_that_end_in_any_warp(oracle_, case):
    """A CTA per block, a sequence per warp: blocks that run out of strings in different warps, often."""
    n, m, l, d = case
    seqs = pi.planted_instance(n, m, l, d, 17).seqs
    want = oracle_.solve_packed(seqs, l, d)
    with pms.Context(0) as c:
        for _ in range(20):
            assert np.array_equal(c.solve(seqs, l, d), want)


# the first: more dense instances than a grid has rows; the second: more than have buckets in one launch
@pytest.mark.parametrize("case", [(66000, 2, 40, 6, 2, 8192), (4200, 3, 456, 7, 2, 131072)], ids=str)
def test_batch_of_many_dense_instances(oracle_, case):
    """Batches whose instances have thousands of motifs each; 33 different instances among them."""
    count, n, m, l, d, cap = case
    kinds = [pi.random_sequences(n, m, 500 + k) for k in range(33)]
    want = [oracle_.solve_packed(s, l, d) for s in kinds]
    assert min(len(w) for w in want) > 1000
    with pms.Context(0) as c:
        c.set_options(max_motifs=cap)
        got = c.solve_batch([(kinds[k % 33], l, d) for k in range(count)])
    assert len(got) == count
    assert all(np.array_equal(g, want[k % 33]) for k, g in enumerate(got))


def _skewed(n, m, p, seed):
    """Sequences whose letters are drawn with the probabilities p."""
    return np.frombuffer(b"ACGT", dtype=np.uint8)[np.random.default_rng(seed).choice(4, size=(n, m), p=p)]


# letters far from uniform: the motifs crowd into few buckets. The first answer's largest bucket is
# within what is ranked bucket by bucket, the second's is not
@pytest.mark.parametrize("p", [(0.8, 0.1, 0.05, 0.05), (0.955, 0.015, 0.015, 0.015)], ids=str)
def test_skewed_letters_match_oracle(oracle_, p):
    seqs = _skewed(12, 700, p, 5)
    want = oracle_.solve_packed(seqs, 11, 3, cap=1 << 26)
    assert len(want) > 8192
    with pms.Context(0) as c:
        for _ in range(3):   # kernel by kernel, captured, replayed
            assert np.array_equal(c.solve(seqs, 11, 3), want)
        for got in c.solve_batch([(seqs, 11, 3)] * 3):
            assert np.array_equal(got, want)


def test_skewed_letters_in_a_large_answer():
    """Five million motifs, 46,000 of them in the fullest bucket (one warp would rank it for 1.8 s); the
    answer is in order, and strings near the sequences are in it exactly if every sequence has them."""
    seqs = _skewed(6, 900, (0.8, 0.1, 0.05, 0.05), 5)
    l, d = 14, 4
    with pms.Context(0) as c:
        c.set_options(graph=-1)
        got = c.solve(seqs, l, d)
        assert c.stats()["ms_kernel"] < 400
    assert len(got) > 1 << 22 and np.all(got[1:] > got[:-1])
    code = np.searchsorted(np.frombuffer(b"ACGT", dtype=np.uint8), seqs)
    windows = np.lib.stride_tricks.sliding_window_view(code, l, axis=1)
    place = 4 ** np.arange(l - 1, -1, -1)
    rng, inside = np.random.default_rng(6), 0
    for _ in range(2000):
        s = windows[rng.integers(6), rng.integers(windows.shape[1])].copy()
        at = rng.permutation(l)[:rng.integers(d + 3)]
        s[at] = rng.integers(0, 4, len(at))
        want = bool(((windows != s).sum(axis=2) <= d).any(axis=1).all())
        key = np.uint64(s @ place)
        i = np.searchsorted(got, key)
        assert (i < len(got) and got[i] == key) == want
        inside += want
    assert 100 < inside < 1900


def test_raw_count_beyond_32_bits():
    """Every one of the 4^10 strings is a motif, and each is near some 4,100 of the 52,428 seed windows:
    the raw count is 52428 |B(10,5)| = 2^32 + 39320."""
    import torch
    n, m, l, d = 2, 52437, 10, 5
    seqs = pi.random_sequences(n, m, 8)
    with pms.Context(0) as c:
        assert np.array_equal(c.solve(seqs, l, d), np.arange(4 ** l, dtype=np.uint64))
        out = torch.zeros(4 ** l, dtype=torch.int64, device="cuda")
        st = torch.zeros(4, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        c.solve_device(torch.from_numpy(seqs.copy()).cuda(), n, m, l, d, out, 4 ** l, st)
        torch.cuda.synchronize()
        assert list(st.cpu().numpy().astype(np.uint32)[:3]) == [0xffffffff, 4 ** l, 2]
        c.set_options(max_motifs=1 << 16)   # above what the count's low 32 bits say
        with pytest.raises(pms.PMSError) as e:
            c.solve(seqs, l, d)
        assert e.value.code == pms.PMS_ETOOMANY


@pytest.mark.parametrize("case", [(20, 1000, 13, 4), (20, 800, 15, 4), (20, 600, 11, 3)], ids=str)
def test_ctas_per_sm_bounds_the_sieve(case):
    """One CTA per multiprocessor: the same motifs, later (but in the form for few blocks, whose 256 CTAs
    are hardly more than one for each)."""
    n, m, l, d = case
    seqs = pi.planted_instance(n, m, l, d, 3).seqs
    got, ms = [], []
    for per_sm in (0, 1):
        with pms.Context(0) as c:
            c.set_options(ctas_per_sm=per_sm, graph=-1)
            times = []
            for _ in range(5):
                got.append(c.solve(seqs, l, d))
                times.append(c.stats()["ms_verify"])
            ms.append(min(times))
    assert all(np.array_equal(g, got[0]) for g in got)
    assert l == 11 or ms[1] > 1.2 * ms[0]


# (n, m, l, d, q, alone) by the form that the runtime takes for them on 152 multiprocessors (test_sieve_forms_host.py
# holds it to that): middle letters, counter planes, warps per block. Windows a sequence at and around the
# multiples of 32 and 256, one window, numbers of sequences around a CTA's warps and what the planes count
# up to, quorums of one, of about half and of all but one.
FORMS = {
    (3, 0, 0): [(2, 10, 6, 1, 2, 1), (3, 8, 8, 1, 3, 1), (7, 36, 6, 2, 7, 1), (8, 39, 8, 3, 8, 1), (20, 41, 9, 2, 20, 1),
                (31, 72, 9, 3, 31, 1), (21, 74, 10, 4, 21, 1)],
    (3, 0, 1): [(21, 10, 6, 2, 21, 0), (2, 260, 6, 1, 2, 0), (3, 38, 8, 3, 3, 0), (9, 41, 10, 3, 9, 0),
                (20, 607, 8, 1, 20, 0), (31, 72, 10, 4, 31, 0)],
    (4, 0, 0): [(2, 11, 11, 2, 2, 1), (3, 15, 11, 3, 3, 1), (7, 41, 11, 4, 7, 1), (8, 42, 11, 5, 8, 1), (9, 43, 11, 2, 9, 1),
                (33, 75, 11, 2, 33, 1)],
    (4, 0, 1): [(3, 11, 11, 6, 3, 0), (2, 15, 11, 5, 2, 0), (8, 41, 11, 4, 8, 0), (9, 43, 12, 4, 9, 0), (20, 44, 12, 5, 20, 0),
                (31, 75, 11, 3, 31, 0)],
    (5, 0, 1): [(8, 18, 14, 6, 8, 0), (7, 77, 13, 4, 7, 0), (3, 45, 14, 5, 3, 1), (9, 45, 13, 5, 9, 0), (21, 270, 14, 4, 21, 0),
                (31, 114, 15, 5, 31, 1), (33, 76, 13, 4, 33, 0)],
    (5, 0, 8): [(2, 12, 12, 1, 2, 1), (7, 17, 13, 2, 7, 1), (9, 44, 12, 3, 9, 1), (3, 43, 13, 4, 3, 1), (8, 43, 12, 4, 8, 1),
                (21, 76, 12, 5, 21, 1), (31, 75, 13, 5, 31, 1)],
    (6, 0, 8): [(2, 268, 14, 1, 2, 1), (3, 269, 14, 4, 3, 0), (7, 413, 14, 1, 7, 1), (20, 268, 14, 1, 20, 1)],
    (3, 7, 1): [(20, 6, 6, 3, 19, 0), (3, 10, 6, 4, 2, 1), (64, 30, 6, 1, 1, 0), (64, 73, 8, 2, 63, 0), (63, 71, 8, 2, 31, 0),
                (9, 134, 6, 2, 4, 0), (32, 262, 8, 1, 16, 0), (33, 70, 11, 3, 30, 0), (31, 69, 6, 2, 1, 1)],
    (4, 5, 1): [(8, 17, 13, 5, 7, 0), (20, 12, 12, 5, 18, 0), (9, 76, 12, 3, 4, 0), (31, 20, 12, 4, 30, 0),
                (21, 44, 12, 4, 10, 1), (31, 76, 14, 4, 15, 1), (20, 77, 14, 5, 10, 0)],
    (5, 5, 8): [(9, 267, 13, 3, 7, 1), (7, 268, 13, 4, 6, 1), (31, 613, 14, 3, 15, 1), (21, 312, 13, 3, 10, 0),
                (31, 400, 13, 3, 30, 1), (20, 269, 14, 5, 19, 1)],
}


@pytest.mark.parametrize("form,case", [(f, c) for f in FORMS for c in FORMS[f]], ids=str)
def test_every_form_at_its_edges(oracle_, form, case):
    """Each kernel of the sieve: against the oracle where that is quick, and against the tree form."""
    n, m, l, d, q, alone = case
    seqs = pi.planted_instance(n, m, l, d, 13).seqs
    with pms.Context(0) as c, pms.Context(0) as tree:
        c.set_options(quorum=q)
        tree.set_options(quorum=q, grab=1)
        want = tree.solve(seqs, l, d)
        assert len(want) > 0
        if l <= 11:
            assert np.array_equal(want, oracle_.solve_quorum(seqs, l, d, q, cap=1 << 24))
        for got in [c.solve(seqs, l, d)] if alone else c.solve_batch([(seqs, l, d)] * 3):
            assert np.array_equal(got, want)
