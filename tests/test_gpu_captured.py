"""Captured graphs -- a run's generations, a caller's own capture -- beside other
calls on the same handle: what a graph points at stays, whatever the handle
does in between."""
import numpy as np
import pytest

import oracle
import paper_1801_03039_gb300 as eb
from helpers import assert_bits_equal, oracle_eval
from test_gpu_ea import BASE, _compare_generation, _device_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    pytest.importorskip("torch")
    eb.build()
    oracle.build()


def matrix(R, C, seed=0):
    return np.random.default_rng(seed).standard_normal((R, C)).astype(np.float32)


def population(rng, P, C, n):
    off = np.arange(0, n * P + 1, n, dtype=np.int32)
    return off, np.concatenate([rng.permutation(C)[:n] for _ in range(P)]).astype(np.int32)


@pytest.mark.parametrize("table", [False, True])
def test_larger_evaluations_between_generations(table):
    """Series of 5,000 rows are split (planes, or table parts of 4,096 rows), in
    the run's generations and in ever larger evaluations between them, both
    counting through counters that the evaluations outgrow."""
    A = matrix(5000, 12)
    kw = {**BASE, "iterations": 22, "pop_size": 60, "sigma": 30, "fitness_support": 1}
    ref = oracle.run(A, trace=True, **kw)
    rng = np.random.default_rng(1)
    h = eb.ebic_load_matrix(A)
    try:
        eb.ebic_set_path(h, eb.PATH_BITMASK if table else eb.PATH_GATHER)
        if table:
            eb.ebic_set_eval_tuning(h, kernel=2, vecs_per_part_bitmask=32)
        eb.ebic_run_init(h, _device_params(kw))
        done = 0
        for step, P in ((2, 100), (3, 3000), (16, 12000), (1, 20)):
            off, cols = population(rng, P, 12, 3)
            inc, dec, fit = oracle_eval(A, off, cols, 30, 1)
            got = eb.ebic_eval_population(h, off, cols, 30, 1)
            for g, w in zip(got, (inc, dec, fit)):
                assert_bits_equal(g, w, P)
            eb.ebic_run_step(h, step)
            done += step
            _compare_generation(h, ref, done, kw["pop_size"], kw["toprank_size"], kw["len_max"], kw)
    finally:
        eb.ebic_free(h)


@pytest.mark.parametrize("table", [False, True])
def test_larger_evaluation_after_a_capture(table):
    """A caller's graph over a split evaluation, replayed after the handle has
    evaluated a population many times as large."""
    import torch
    A = matrix(9000, 20, 2)
    rng = np.random.default_rng(3)
    h = eb.ebic_load_matrix(A)
    try:
        if table:
            eb.ebic_build_pair_table(h)
            eb.ebic_set_eval_tuning(h, kernel=2, vecs_per_part_bitmask=32)
        off, cols = population(rng, 50, 20, 4)
        want = oracle_eval(A, off, cols, 9, 1)
        d_off, d_cols = torch.from_numpy(off).cuda(), torch.from_numpy(cols).cuda()
        inc = torch.zeros(50, dtype=torch.int32, device="cuda")
        dec, fit = torch.zeros_like(inc), torch.zeros(50, dtype=torch.float64, device="cuda")

        def evaluate(stream):
            eb.ebic_eval_population_dev(h, d_off, d_cols, 50, len(cols), 9, 1, inc, dec, fit, stream)

        s = torch.cuda.Stream()
        evaluate(s)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            evaluate(torch.cuda.current_stream())
        for P in (4000, 15000):
            o, c = population(rng, P, 20, 3)
            got = eb.ebic_eval_population(h, o, c, 9, 1)
            assert_bits_equal(got[0], oracle_eval(A, o, c, 9, 1)[0], P)
            for t in (inc, dec, fit):
                t.fill_(-1)
            graph.replay()
            torch.cuda.synchronize()
            eb.ebic_check_device_error(h)
            assert_bits_equal(inc.cpu().numpy().view(np.uint32), want[0], "inc")
            assert_bits_equal(dec.cpu().numpy().view(np.uint32), want[1], "dec")
            assert_bits_equal(fit.cpu().numpy(), want[2], "fitness")
    finally:
        eb.ebic_free(h)


def test_smaller_run_beside_a_larger_one():
    """Two handles: a run that needs much shared memory goes on, by replays and
    by separate launches, after a run that needs little has started."""
    A = matrix(300, 200, 4)
    kw = {**BASE, "iterations": 22, "pop_size": 2048, "len_min": 3, "len_max": 60, "sigma": 5,
          "toprank_size": 1000}
    ref = oracle.run(A, trace=True, **kw)
    large, small = eb.ebic_load_matrix(A), eb.ebic_load_matrix(A[:, :140].copy())
    try:
        eb.ebic_run_init(large, _device_params(kw))
        eb.ebic_run_init(small, _device_params({**BASE, "pop_size": 20, "toprank_size": 20,
                                                "len_max": 4}))
        done = 0
        for step in (0, 1, 20):
            if step:
                eb.ebic_run_step(large, step)
            else:
                eb.ebic_run_step_profiled(large)
            done += step or 1
            _compare_generation(large, ref, done, kw["pop_size"], kw["toprank_size"],
                                kw["len_max"], kw)
    finally:
        eb.ebic_free(large)
        eb.ebic_free(small)


def test_both_counts_without_a_falling_output():
    """Fitness over rising and falling rows, falling counts not asked for: a
    captured call and a larger one after it share no scratch."""
    import torch
    A = matrix(3000, 20, 5)
    rng = np.random.default_rng(6)
    h = eb.ebic_load_matrix(A)
    try:
        def call(P, n):
            off, cols = population(rng, P, 20, n)
            inc, _, fit = oracle_eval(A, off, cols, 9, 1)
            d = [torch.from_numpy(off).cuda(), torch.from_numpy(cols).cuda(),
                 torch.zeros(P, dtype=torch.int32, device="cuda"),
                 torch.zeros(P, dtype=torch.float64, device="cuda")]

            def run(stream):
                eb.ebic_eval_population_dev(h, d[0], d[1], P, len(cols), 9, 1, d[2], None, d[3],
                                            stream)

            def check(what):
                torch.cuda.synchronize()
                assert_bits_equal(d[2].cpu().numpy().view(np.uint32), inc, (what, "inc"))
                assert_bits_equal(d[3].cpu().numpy(), fit, (what, "fitness"))
                d[2].fill_(-1)
                d[3].fill_(-1)

            return run, check

        s = torch.cuda.Stream()
        for table in (False, True):
            if table:
                eb.ebic_build_pair_table(h)
            run, check = call(50, 4)
            run(s)
            check("first")
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=s):
                run(torch.cuda.current_stream())
            run2, check2 = call(6000, 3)
            run2(s)
            check2("larger")
            graph.replay()
            check("replayed")
    finally:
        eb.ebic_free(h)


@pytest.mark.parametrize("C", [200, 600])
def test_host_calls_and_runs_behind_a_table_being_built(C):
    """The table built on the caller's stream and not waited for, right before a
    call with host buffers and a run, which work on the handle's own stream."""
    import torch
    A = matrix(30000, C, 7)
    rng = np.random.default_rng(9)
    off, cols = population(rng, 300, C, 4)
    want = oracle_eval(A, off, cols, 9)
    kw = {**BASE, "iterations": 2, "sigma": 9}
    ref = oracle.run(A, trace=True, **kw)
    for stream in (None, torch.cuda.Stream()):
        for run in (False, True):
            h = eb.ebic_load_matrix(A)
            try:
                eb.ebic_build_pair_table(h, stream)
                if run:
                    eb.ebic_run_init(h, _device_params(kw))
                    eb.ebic_run_step(h, 2)
                    _compare_generation(h, ref, 2, kw["pop_size"], kw["toprank_size"],
                                        kw["len_max"], kw)
                for g, w in zip(eb.ebic_eval_population(h, off, cols, 9), want):
                    assert_bits_equal(g, w, (stream, run))
            finally:
                torch.cuda.synchronize()
                eb.ebic_free(h)


@pytest.mark.parametrize("calls", [(150,), (127, 1, 16, 6), (60, 60, 30), (10,) * 15])
def test_generations_of_a_long_run(calls):
    """Runs that reach the 128 generations from which they are replayed sixteen to a
    graph, in one call or several, with an evaluation that outgrows the handle's
    counters between the calls; and one that stops in the middle of such a graph."""
    rng = np.random.default_rng(11)
    for A, kw in ((matrix(2000, 20, 8), dict(iterations=150, sigma=20)),
                  (matrix(50, 3, 9), dict(iterations=150, pop_size=6, len_min=2, len_max=3, sigma=2,
                                          toprank_size=10))):
        kw = {**BASE, **kw}
        ref = oracle.run(A, trace=True, **kw)
        h = eb.ebic_load_matrix(A)
        try:
            eb.ebic_set_path(h, eb.PATH_GATHER)          # 2,000 rows: split series
            eb.ebic_run_init(h, _device_params(kw))
            done, P = 0, 150
            for n in calls:
                stats = eb.ebic_run_step(h, n)
                done += n
                if stats["stop_reason"] == 0:
                    _compare_generation(h, ref, done, kw["pop_size"], kw["toprank_size"],
                                        kw["len_max"], kw)
                P = min(2 * P, 10000)
                off, cols = population(rng, P, A.shape[1], 2)
                assert_bits_equal(eb.ebic_eval_population(h, off, cols, 3)[0],
                                  oracle_eval(A, off, cols, 3)[0], P)
            for key in ("generations_done", "stop_reason", "tabu_hits_total", "attempts_total",
                        "toprank_n"):
                assert stats[key] == ref["stats"][key], key
            assert eb.ebic_get_toprank(h, kw["toprank_size"], kw["len_max"])[0] == ref["toprank"]
        finally:
            eb.ebic_free(h)


def test_run_whose_surrogate_was_released():
    """A surrogate can be freed once detached; the run that screened with it is still
    there to be read, and refuses every kind of step until it is started again."""
    A = matrix(300, 40, 14)
    h = eb.ebic_load_matrix(A)
    try:
        s = eb.ebic_surrogate_create(h, 8, 3)
        eb.ebic_run_screen(h, s, 4, eb.SCREEN_SURROGATE)
        p = eb.ebic_default_params(pop_size=50, iterations=20, sigma=5)
        eb.ebic_run_init(h, p)
        eb.ebic_run_step(h, 2)
        top = eb.ebic_get_toprank(h, 100, 6)[0]
        with pytest.raises(eb.EbicError):
            eb.ebic_surrogate_free(s)
        eb.ebic_run_screen(h, None, 1, eb.SCREEN_OFF)
        eb.ebic_run_step(h, 0)                            # detached, not freed
        eb.ebic_surrogate_free(s)
        for step in (lambda: eb.ebic_run_step(h, 1), lambda: eb.ebic_run_step_async(h, 1),
                     lambda: eb.ebic_run_step_profiled(h)):
            with pytest.raises(eb.EbicError) as e:
                step()
            assert e.value.status == 5                    # EBIC_ERR_STATE
        assert eb.ebic_run_step(h, 0)["generations_done"] == 2
        assert eb.ebic_get_toprank(h, 100, 6)[0] == top
        eb.ebic_run_init(h, p)
        assert eb.ebic_run_step(h, 3)["generations_done"] == 3
    finally:
        eb.ebic_free(h)
