"""The generation loop, surrogate training and batched evaluation at the edges
of their kernels' tiles, batches and buffers."""
import numpy as np
import pytest

import oracle
import paper_1801_03039_gb300 as eb
from oracle import mlp
from helpers import assert_bits_equal, oracle_eval
from test_gpu_ea import BASE, _compare_generation, _device_params, run_both
from test_gpu_surrogate import _device_series, _oracle_params, _series

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    pytest.importorskip("torch")
    eb.build()
    oracle.build()


def matrix(R, C, seed=0):
    return np.random.default_rng(seed).standard_normal((R, C)).astype(np.float32)


# ---- Steps 1-5 ----

@pytest.mark.parametrize("C,len_max", [(4, 3), (127, 6), (128, 7), (129, 6), (255, 7), (256, 6),
                                       (257, 6), (100, 33), (90, 64)])
def test_search_at_the_bitset_widths(C, len_max):
    """Columns at the edges of four and eight words (257: the general path);
    even and odd row strides; entrants of more columns than the builder holds
    in registers (two halves of sixteen)."""
    run_both(matrix(60, C), iterations=4, len_max=len_max, len_min=2, sigma=4,
             pop_size=12 if C == 4 else 150)


@pytest.mark.parametrize("k", [1, 2])
@pytest.mark.parametrize("P", [2, 15, 16, 31, 32, 33, 63, 65])
def test_search_at_the_batch_edges(P, k):
    """2 P + 1 attempts at the edges of batches of 32 and of the buffers' ring."""
    run_both(matrix(80, 20), iterations=6, pop_size=P, tournament_k=k, toprank_size=7)


def test_generations_of_one_call():
    """One call's generations, most of them sixteen to a graph, against the
    oracle, and a run that stops in the middle of such a graph."""
    for A, kw in ((matrix(200, 20), dict(iterations=53)),
                  (matrix(50, 3), dict(iterations=100, pop_size=6, len_min=2, len_max=3, sigma=2,
                                       toprank_size=10))):
        kw = {**BASE, **kw}
        ref = oracle.run(A, trace=True, **kw)
        h = eb.ebic_load_matrix(A)
        try:
            eb.ebic_run_init(h, _device_params(kw))
            stats = eb.ebic_run_step(h, kw["iterations"])
            for key in ("generations_done", "stop_reason", "tabu_hits_total", "attempts_total",
                        "toprank_n"):
                assert stats[key] == ref["stats"][key], key
            if stats["stop_reason"] == 0:
                _compare_generation(h, ref, kw["iterations"], kw["pop_size"], kw["toprank_size"],
                                    kw["len_max"], kw)
            top, fit, _ = eb.ebic_get_toprank(h, kw["toprank_size"], kw["len_max"])
            assert top == ref["toprank"]
            assert_bits_equal(fit, ref["toprank_f"], "toprank fitness")
        finally:
            eb.ebic_free(h)


@pytest.mark.parametrize("C,P,T,tau", [(20, 400, 400, 1.0), (20, 400, 400, 0.0), (200, 64, 2, 0.3),
                                       (250, 2500, 2500, 1.0)])
def test_list_room(C, P, T, tau):
    """Step 5 where all individuals join (the last case outgrows the shared
    room, so the CTA-wide kernel stands in), where any overlap evicts, and with
    fewer records kept than one window tests."""
    run_both(matrix(60, C), iterations=3, pop_size=P, toprank_size=T, overlap_tau=tau, sigma=4)


# ---- surrogate training ----

def _grads(h, kind, flat, batches, seed=4, S=20):
    s = eb.ebic_surrogate_create(h, S, seed)
    try:
        eb.ebic_surrogate_train_kernel(s, kind)
        eb.ebic_surrogate_params(s, flat)
        for d_seq, d_len, d_t, B in batches:
            loss = eb.ebic_surrogate_step(s, d_seq, d_len, S, d_t, B, update=False)
        return loss, eb.ebic_surrogate_grads(s)
    finally:
        eb.ebic_surrogate_free(s)


@pytest.mark.parametrize("C,B", [(100, 1), (100, 2), (60, 127), (200, 128), (201, 129), (300, 257),
                                 (100, 20000)])
def test_training_tiles(C, B):
    """Minibatches at the edges of the 128-row tile, of more tiles than SMs, and
    columns at the edges of the embedding's segments.  The two training kernels
    round at the same points; sums in another order can flip roundings of dh2,
    dh1 and h by one bf16 unit (2^-8 each), below 2^-6 together.  A smaller
    minibatch after a larger one gives the bits of a fresh surrogate."""
    import torch
    h = eb.ebic_load_matrix(matrix(300, C, 3))
    try:
        _, flat = _oracle_params(C, 13)
        rng = np.random.default_rng(B)

        def minibatch(n):
            d_seq, d_len = _device_series(_series(rng, n, C, 1, 20), 20)
            return d_seq, d_len, torch.from_numpy(rng.standard_normal(n).astype(np.float32) - 5).cuda(), n

        one, larger = minibatch(B), minibatch(B + 140)
        la, ga = _grads(h, eb.FORWARD_TCGEN05, flat, [one])
        lb, gb = _grads(h, eb.FORWARD_MMA_SYNC, flat, [one])
        assert abs(la - lb) <= 1e-3 * abs(lb)
        sa, sb = (eb.ebic_surrogate_split(g.astype(np.float64), C) for g in (ga, gb))
        for name in sa:
            a, b = np.asarray(sa[name]).reshape(-1), np.asarray(sb[name]).reshape(-1)
            assert np.linalg.norm(a - b) <= 2 ** -6 * np.linalg.norm(b), name
        for kind in (eb.FORWARD_TCGEN05, eb.FORWARD_MMA_SYNC):
            want = _grads(h, kind, flat, [one])
            got = _grads(h, kind, flat, [larger, one])
            assert got[0] == want[0]
            assert_bits_equal(got[1], want[1], "gradients after a larger minibatch")
    finally:
        eb.ebic_free(h)


# ---- batched evaluation ----

@pytest.mark.parametrize("tables", ["none", "some", "all"])
def test_batch_of_uneven_items(tables):
    """Problems of one row to many parts, with and without pair tables side by
    side, series of up to 100 columns (repeats allowed), and an invalid column in
    one problem, whose series counts nothing while the others' results stand."""
    import torch
    rng = np.random.default_rng(7)
    shapes = [(1, 3, 1), (31, 40, 33), (129, 2, 5), (4097, 120, 400), (40000, 60, 257), (70000, 9, 3)]
    handles, items, want, outs = [], [], [], []
    try:
        for k, (R, C, P) in enumerate(shapes):
            A = matrix(R, C, k)
            seqs = [rng.integers(0, C, int(rng.choice([1, 2, 5, 31, 33, 100]))) for _ in range(P)]
            off = np.cumsum([0] + [len(s) for s in seqs]).astype(np.int32)
            cols = np.concatenate(seqs).astype(np.int32)
            h = eb.ebic_load_matrix(A)
            handles.append(h)
            if tables == "all" or (tables == "some" and k % 2):
                eb.ebic_build_pair_table(h)
            inc, _, fit = oracle_eval(A, off, cols, 5)
            if k == 3:
                cols[off[7]] = C
                inc[7], fit[7] = 0, 0.0
            want.append((inc, fit))
            o = (torch.full((P,), -1, dtype=torch.int32, device="cuda"),
                 torch.full((P,), -1.0, dtype=torch.float64, device="cuda"))
            outs.append(o)
            items.append((torch.from_numpy(off).cuda(), torch.from_numpy(cols).cuda(), P, len(cols), 5) + o)
        b = eb.ebic_batch_create(handles, items, 0)
        try:
            for _ in range(2):
                for inc, fit in outs:
                    inc.fill_(-1)
                    fit.fill_(-1.0)
                eb.ebic_batch_eval(b)
                torch.cuda.synchronize()
                for k, (inc, fit) in enumerate(outs):
                    if k == 3:
                        with pytest.raises(eb.EbicError):
                            eb.ebic_check_device_error(handles[k])
                    else:
                        eb.ebic_check_device_error(handles[k])
                    assert_bits_equal(inc.cpu().numpy().view(np.uint32), want[k][0], f"inc {k}")
                    assert_bits_equal(fit.cpu().numpy(), want[k][1], f"fitness {k}")
        finally:
            eb.ebic_batch_free(b)
    finally:
        for h in handles:
            eb.ebic_free(h)


# ---- evaluation ----

@pytest.mark.parametrize("R", [4096, 20000, 70000])
def test_split_series_with_both_counts(R):
    """Rising and falling counts of series split over parts: one word of a
    handle's counters holds both and the arrivals."""
    A = matrix(R, 12)
    A[::50] = np.nan
    rng = np.random.default_rng(R)
    seqs = [rng.permutation(12)[:int(rng.integers(1, 7))] for _ in range(90)]
    off = np.cumsum([0] + [len(s) for s in seqs]).astype(np.int32)
    cols = np.concatenate(seqs).astype(np.int32)
    inc, dec, fit = oracle_eval(A, off, cols, 3, 1)
    h = eb.ebic_load_matrix(A)
    try:
        eb.ebic_build_pair_table(h)
        for part in (0, 32, 64):
            eb.ebic_set_eval_tuning(h, vecs_per_part_bitmask=part)
            for _ in range(2):
                g = eb.ebic_eval_population(h, off, cols, 3, 1, want_dec=True)
                assert_bits_equal(g[0], inc, ("inc", part))
                assert_bits_equal(g[1], dec, ("dec", part))
                assert_bits_equal(g[2], fit, ("fitness", part))
    finally:
        eb.ebic_free(h)


@pytest.mark.parametrize("P", [21887, 21888])
def test_large_populations_without_table(P):
    """The populations that end the rank planes' range over one slice."""
    rng = np.random.default_rng(P)
    A = matrix(1100, 20)
    off = np.arange(0, 3 * P + 1, 3, dtype=np.int32)
    cols = rng.integers(0, 20, 3 * P).astype(np.int32)
    inc, dec, fit = oracle_eval(A, off, cols, 3)
    h = eb.ebic_load_matrix(A)
    try:
        g = eb.ebic_eval_population(h, off, cols, 3, 0, want_dec=True)
        for got, want in zip(g, (inc, dec, fit)):
            assert_bits_equal(got, want, P)
    finally:
        eb.ebic_free(h)
