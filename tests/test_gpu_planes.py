"""The rank planes on a GPU: the pair table built from them and the evaluation
without a table, against the oracle and numpy, at the edges of their tiles."""
import numpy as np
import pytest

import oracle
from helpers import assert_bits_equal, oracle_eval

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eb():
    import paper_1801_03039_gb300 as m
    m.build()
    oracle.build()
    return m


def awkward(rng, R, C):
    """Ties, both zeros, infinities, subnormals and NaN among normal draws."""
    A = rng.standard_normal((R, C)).astype(np.float32)
    pick = rng.random((R, C))
    A[pick < 0.25] = np.round(A[pick < 0.25])
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-45, -1e-45, np.nan], np.float32)
    odd = pick > 0.93
    A[odd] = special[rng.integers(0, len(special), int(odd.sum()))]
    return A


def population(rng, P, C, long=()):
    seqs = [rng.permutation(C)[:int(rng.integers(1, min(C, 9) + 1))] for _ in range(P)]
    seqs += [rng.integers(0, C, n) for n in long]                 # repeated columns allowed
    off = np.cumsum([0] + [len(s) for s in seqs]).astype(np.int32)
    return off, np.concatenate(seqs).astype(np.int32)


# columns at the edges of the plane counts (6: 63 | 64, 7: 127 | 128, 8: 255 |
# 256, 9: 511; 512 has no planes), rows at the edges of a word, a 16-byte
# vector and a slice (1,024 and 2,048 rows)
SHAPES = [(1, 1), (5, 4), (31, 2), (33, 63), (127, 64), (128, 20), (129, 127), (1000, 128),
          (1024, 100), (1025, 255), (2049, 33), (4097, 256), (700, 511), (700, 512), (9000, 90)]


@pytest.mark.parametrize("R,C", SHAPES)
def test_pair_table_from_planes(eb, R, C):
    rng = np.random.default_rng(R * 1000 + C)
    A = awkward(rng, R, C)
    h = eb.ebic_load_matrix(A)
    try:
        eb.ebic_build_pair_table(h)
        W = (R + 127) // 128 * 4
        pairs = {(0, 0), (0, C - 1), (C - 1, 0), (C - 1, C - 1)}
        pairs |= {tuple(int(v) for v in rng.integers(0, C, 2)) for _ in range(40)}
        row = np.arange(32 * W).reshape(-1, 32, 4).transpose(0, 2, 1).reshape(W, 32)
        for p, q in pairs:
            lt = np.zeros(32 * W, bool)
            lt[:R] = A[:, p] < A[:, q]
            want = (lt[row].astype(np.uint64) << np.arange(32, dtype=np.uint64)).sum(1)
            assert_bits_equal(eb.ebic_read_pair_words(h, p, q, 0, W), want.astype(np.uint32), (p, q))
    finally:
        eb.ebic_free(h)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("R,C", SHAPES)
def test_evaluation_without_table(eb, R, C, mode):
    rng = np.random.default_rng(R * 1000 + C + 7)
    A = awkward(rng, R, C)
    h = eb.ebic_load_matrix(A)
    try:
        for P, long in ((1, ()), (70, (32, 33, 34, 64, 65, 1024)), (2600, ())):
            off, cols = population(rng, P, C, long)
            inc, dec, fit = oracle_eval(A, off, cols, 3, mode)
            for want_dec in (True, False):
                for part in (0, 32):                  # rank planes, then the fp32 columns
                    eb.ebic_set_eval_tuning(h, vecs_per_part_gather=part)
                    g = eb.ebic_eval_population(h, off, cols, 3, mode, want_dec=want_dec)
                    assert_bits_equal(g[0], inc, ("inc", P, part))
                    if want_dec:
                        assert_bits_equal(g[1], dec, ("dec", P, part))
                    assert_bits_equal(g[2], fit, ("fitness", P, part))
    finally:
        eb.ebic_free(h)


def test_bad_columns_without_table(eb):
    """An out-of-range column found on the device: zeros and the error flag."""
    import torch
    rng = np.random.default_rng(5)
    h = eb.ebic_load_matrix(rng.standard_normal((3000, 40)).astype(np.float32))
    try:
        off = torch.tensor([0, 3, 6, 9], dtype=torch.int32, device="cuda")
        cols = torch.tensor([1, 2, 3, 4, 40, 6, 7, -1, 9], dtype=torch.int32, device="cuda")
        inc = torch.full((3,), 9, dtype=torch.int32, device="cuda")
        fit = torch.full((3,), 9.0, dtype=torch.float64, device="cuda")
        eb.ebic_eval_population_dev(h, off, cols, 3, 9, 5, eb.SUPPORT_INC, inc, None, fit)
        with pytest.raises(eb.EbicError):
            eb.ebic_check_device_error(h)
        assert inc.tolist()[1:] == [0, 0] and fit.tolist()[1:] == [0.0, 0.0]
        assert inc[0] > 0
    finally:
        eb.ebic_free(h)


@pytest.mark.parametrize("R,C", SHAPES)
def test_rows_from_planes(eb, R, C):
    """Steps 6-7 at the edges of a word, vector and slice; break counts at the
    edges of the counters' widths (2, 4 and 11 bits)."""
    rng = np.random.default_rng(R * 1000 + C + 13)
    A = awkward(rng, R, C)
    h = eb.ebic_load_matrix(A)
    try:
        off, cols = population(rng, 40, C, (33, 64, 300))
        seqs = [cols[off[i]:off[i + 1]] for i in range(len(off) - 1)]
        for mode in (0, 1):
            got = eb.ebic_extract_rows(h, off, cols, mode)
            for s, g in zip(seqs, got):
                assert g.dtype == np.int32 and g.tolist() == list(oracle.rows(A, s, mode))
            for e in (0, 1, 3, 4, 15, 16, 1024):
                got = eb.ebic_extract_rows_approx(h, off, cols, e, mode)
                for s, g in zip(seqs, got):
                    assert g.tolist() == list(oracle.rows_approx(A, s, e, mode)), (e, mode)
    finally:
        eb.ebic_free(h)


def test_rows_of_more_than_the_first_guess(eb):
    """More rows than the binding offers at first, and than the handle's buffer."""
    R = 30000
    A = np.random.default_rng(3).standard_normal((R, 8)).astype(np.float32)
    h = eb.ebic_load_matrix(A)
    try:
        for P in (2, 40, 3):
            off = np.arange(P + 1, dtype=np.int32)
            rows = eb.ebic_extract_rows(h, off, np.arange(P, dtype=np.int32) % 8)
            assert len(rows) == P and all(np.array_equal(r, np.arange(R)) for r in rows)
    finally:
        eb.ebic_free(h)
