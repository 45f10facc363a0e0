"""The rank planes are made by the first call that reads them: what a handle that
was only loaded holds, and evaluations, tables and rows in every order, on other
streams and under capture."""
import numpy as np
import pytest

import oracle
import paper_1801_03039_gb300 as eb
from helpers import assert_bits_equal, oracle_eval

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    pytest.importorskip("torch")
    eb.build()
    oracle.build()


def test_a_loaded_matrix_holds_no_planes():
    import torch
    R, C = 100000, 500
    A = torch.randn(R, C, device="cuda")
    eb.ebic_free(eb.ebic_load_matrix_dev(A))             # whatever a first load sets up
    free = torch.cuda.mem_get_info()[0]
    h = eb.ebic_load_matrix_dev(A)
    try:
        used = free - torch.cuda.mem_get_info()[0]
        # columns padded to 128 rows, 2 R + 2 logs, and the driver's 2 MB granularity;
        # the planes would be 56 MB
        assert used <= 4 * C * (R + 127) + 8 * (2 * R + 2) + (8 << 20)
    finally:
        eb.ebic_free(h)


@pytest.mark.parametrize("R,C", [(1000, 20), (5000, 300)])
@pytest.mark.parametrize("order", ["eval table eval", "table eval rows", "rows table eval",
                                   "rows eval table", "eval rows"])
def test_orders_of_first_use(R, C, order):
    """Each call on another stream than the one before, none waited for but by
    its own results."""
    import torch
    rng = np.random.default_rng(R + C)
    A = rng.standard_normal((R, C)).astype(np.float32)
    A[::40] = np.nan
    seqs = [rng.permutation(C)[:int(rng.integers(1, 6))] for _ in range(70)]
    off = np.cumsum([0] + [len(s) for s in seqs]).astype(np.int32)
    cols = np.concatenate(seqs).astype(np.int32)
    inc, dec, fit = oracle_eval(A, off, cols, 5)
    d = [torch.from_numpy(v).cuda() for v in (off, cols)]
    out = [torch.zeros(70, dtype=t, device="cuda") for t in (torch.int32, torch.int32, torch.float64)]
    h = eb.ebic_load_matrix(A)
    try:
        eb.ebic_set_path(h, eb.PATH_GATHER)
        for what in order.split():
            s = torch.cuda.Stream()
            if what == "table":
                eb.ebic_build_pair_table(h, s)
            elif what == "rows":
                for q, rows in zip(seqs, eb.ebic_extract_rows(h, off, cols, 1)):
                    assert rows.tolist() == list(oracle.rows(A, q, 1))
            else:
                eb.ebic_eval_population_dev(h, d[0], d[1], 70, len(cols), 5, 0, *out, s)
                s.synchronize()
                for got, want in zip(out, (inc, dec, fit)):
                    assert_bits_equal(got.cpu().numpy().view(want.dtype), want, what)
                    got.fill_(-1)
                torch.cuda.synchronize()
        if "table" in order:
            torch.cuda.synchronize()
            eb.ebic_set_path(h, eb.PATH_BITMASK)
            got = eb.ebic_eval_population(h, off, cols, 5)
            for g, want in zip(got, (inc, dec, fit)):
                assert_bits_equal(g, want, "table")
    finally:
        eb.ebic_free(h)


def test_a_first_call_under_capture():
    """Up to 1,024 rows an evaluation without a table needs no scratch: its first
    call can be captured, before the handle has planes, and the graph stands after
    it has them."""
    import torch
    rng = np.random.default_rng(8)
    A = rng.standard_normal((1000, 30)).astype(np.float32)
    off = np.arange(0, 303, 3, dtype=np.int32)
    cols = rng.integers(0, 30, 300).astype(np.int32)
    want = oracle_eval(A, off, cols, 5)
    d = [torch.from_numpy(v).cuda() for v in (off, cols)]
    out = [torch.zeros(100, dtype=t, device="cuda") for t in (torch.int32, torch.int32, torch.float64)]
    h = eb.ebic_load_matrix(A)
    try:
        s = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            eb.ebic_eval_population_dev(h, d[0], d[1], 100, 300, 5, 0, *out,
                                        torch.cuda.current_stream())
        for _ in range(2):
            graph.replay()
            torch.cuda.synchronize()
            for got, w in zip(out, want):
                assert_bits_equal(got.cpu().numpy().view(w.dtype), w, "replay")
                got.fill_(-1)
            for got, w in zip(eb.ebic_eval_population(h, off, cols, 5), want):
                assert_bits_equal(got, w, "call")
    finally:
        eb.ebic_free(h)


@pytest.mark.parametrize("R", [100, 1500])
@pytest.mark.parametrize("P", [1, 1023, 1024, 1025, 2048, 5000])
def test_rows_of_many_series(R, P):
    """Series at the edges of the 1,024 whose offsets one CTA sums, of one slice and
    of two, with one- and two-column series among them."""
    rng = np.random.default_rng(R + P)
    A = rng.standard_normal((R, 9)).astype(np.float32)
    seqs = [rng.permutation(9)[:int(rng.integers(1, 5))] for _ in range(P)]
    off = np.cumsum([0] + [len(s) for s in seqs]).astype(np.int32)
    h = eb.ebic_load_matrix(A)
    try:
        got = eb.ebic_extract_rows(h, off, np.concatenate(seqs).astype(np.int32))
    finally:
        eb.ebic_free(h)
    assert len(got) == P
    for s, g in zip(seqs, got):
        keep = np.ones(R, bool)
        for a, b in zip(s, s[1:]):
            keep &= A[:, a] < A[:, b]
        assert np.array_equal(g, np.flatnonzero(keep))


def test_rows_keep_no_large_workspace():
    """Masks of 50 MB, then a list of 80 MB: neither stays with the handle, nor
    after a call that only asks for the size."""
    import torch
    R = 1 << 20
    rng = np.random.default_rng(4)
    h = eb.ebic_load_matrix_dev(torch.randn(R, 20, device="cuda"))
    try:
        off = np.arange(0, 401 * 7, 7, dtype=np.int32)
        cols = np.concatenate([rng.permutation(20)[:7] for _ in range(400)]).astype(np.int32)
        eb.ebic_extract_rows(h, off[:2], cols[:7])       # what any call keeps
        free = torch.cuda.mem_get_info()[0]
        n = sum(len(r) for r in eb.ebic_extract_rows(h, off, cols))
        assert 0 < n < 400 * R / 1000
        one = np.arange(21, dtype=np.int32)
        assert all(len(r) == R for r in eb.ebic_extract_rows(h, one, one[:20]))
        assert free - torch.cuda.mem_get_info()[0] <= 3 * (32 << 20)
    finally:
        eb.ebic_free(h)


@pytest.mark.parametrize("max_breaks", [None, 1])
def test_rows_without_planes(max_breaks):
    """Lists that grow and shrink between calls, from the fp32 columns (600 of them):
    the calls share the handle's workspaces with each other and with evaluations."""
    R, C = 5000, 600
    rng = np.random.default_rng(5)
    A = rng.standard_normal((R, C)).astype(np.float32)
    h = eb.ebic_load_matrix(A)
    try:
        for P, n in ((3, 4), (60, 1), (200, 3), (1, 2)):
            off = np.arange(0, P * n + 1, n, dtype=np.int32)
            cols = np.concatenate([rng.permutation(C)[:n] for _ in range(P)]).astype(np.int32)
            if max_breaks is None:
                got = eb.ebic_extract_rows(h, off, cols, 1)
            else:
                got = eb.ebic_extract_rows_approx(h, off, cols, max_breaks, 1)
            assert len(got) == P
            for i, g in enumerate(got):
                s = cols[off[i]:off[i + 1]]
                want = oracle.rows(A, s, 1) if max_breaks is None else oracle.rows_approx(A, s, 1, 1)
                assert g.tolist() == list(want)
            inc, dec, fit = oracle_eval(A, off, cols, 5)
            for g, w in zip(eb.ebic_eval_population(h, off, cols, 5), (inc, dec, fit)):
                assert_bits_equal(g, w, P)
    finally:
        eb.ebic_free(h)


def test_planes_come_with_use():
    """A matrix of 300 columns gets its planes with the call that brings the series
    evaluated from the columns to C^2 / 20 = 4,500 (a series extracted counts as 12):
    one launch more, the same results before and after."""
    rng = np.random.default_rng(12)
    R, C, P = 3000, 300, 1000
    A = rng.standard_normal((R, C)).astype(np.float32)
    A[::30] = np.nan
    off = np.arange(0, 4 * P + 1, 4, dtype=np.int32)
    cols = np.concatenate([rng.permutation(C)[:4] for _ in range(P)]).astype(np.int32)
    want = oracle_eval(A, off, cols, 5)
    h = eb.ebic_load_matrix(A)
    try:
        eb.ebic_set_path(h, eb.PATH_GATHER)
        launched = []
        for k in range(7):
            before = eb.ebic_kernel_launches()
            if k == 1:                                  # 50 series: 600
                for i, g in enumerate(eb.ebic_extract_rows(h, off[:51], cols[:200], 1)):
                    assert g.tolist() == list(oracle.rows(A, cols[4 * i:4 * i + 4], 1))
                continue
            for g, w in zip(eb.ebic_eval_population(h, off, cols, 5), want):
                assert_bits_equal(g, w, k)
            launched.append(eb.ebic_kernel_launches() - before)
        assert launched == [1, 1, 1, 2, 1, 1]           # 1,000 1,600 2,600 3,600 4,600
    finally:
        eb.ebic_free(h)


@pytest.mark.parametrize("tuned", [False, True])
def test_a_search_without_a_table_has_planes(tuned):
    """At its start, whatever its size: its generations are captured once."""
    from test_gpu_ea import BASE, _compare_generation, _device_params
    A = np.random.default_rng(13).standard_normal((1500, 300)).astype(np.float32)
    kw = {**BASE, "iterations": 3, "sigma": 20, "pop_size": 30}
    ref = oracle.run(A, trace=True, **kw)
    h = eb.ebic_load_matrix(A)
    try:
        eb.ebic_set_path(h, eb.PATH_GATHER)
        if tuned:
            eb.ebic_set_eval_tuning(h, kernel=2)
        eb.ebic_run_init(h, _device_params(kw))
        eb.ebic_run_step(h, 3)
        _compare_generation(h, ref, 3, 30, kw["toprank_size"], kw["len_max"], kw)
        before = eb.ebic_kernel_launches()
        eb.ebic_extract_rows(h, [0, 2], [1, 2])
        assert eb.ebic_kernel_launches() - before >= 2   # masks and offsets: from planes
    finally:
        eb.ebic_free(h)
