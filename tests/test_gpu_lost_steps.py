"""A training step whose bounded device wait expired.  The word in which the
kernels report that is set by hand here: no wait is made to expire."""
import ctypes

import numpy as np
import pytest

import paper_1801_03039_gb300 as eb
from helpers import assert_bits_equal

pytestmark = pytest.mark.gpu
C, S, N = 40, 8, 500


class _Word:
    def __init__(self, ptr):
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": (1,), "typestr": "<i4",
                                         "version": 3}


def lost_word(s, name="ebic_internal_lost_word"):
    import torch
    f = getattr(eb.lib(), name)
    f.argtypes, f.restype = [ctypes.c_void_p], ctypes.c_void_p
    return torch.as_tensor(_Word(f(s)), device="cuda")


@pytest.mark.parametrize("kind", [eb.FORWARD_TCGEN05, eb.FORWARD_MMA_SYNC])
@pytest.mark.parametrize("steps", [0, 1, 2, 5, 20])
def test_lost_step(kind, steps):
    """A lost step ends its call with EBIC_ERR_TIMEOUT and changes nothing, at any
    length of the call (queued steps, replays, eight to a graph; 0: one step on
    explicit targets); the next calls go on as if it had not been asked for."""
    torch = pytest.importorskip("torch")
    eb.build()
    rng = np.random.default_rng(2)
    seq = torch.from_numpy(np.argsort(rng.random((N, C)), 1)[:, :S].astype(np.int16)).cuda()
    length = torch.from_numpy(rng.integers(1, S + 1, N).astype(np.int32)).cuda()
    fit = torch.from_numpy(rng.random(N) * 100).cuda()
    target = torch.from_numpy(rng.standard_normal(N).astype(np.float32)).cuda()
    h = eb.ebic_load_matrix(rng.standard_normal((300, C)).astype(np.float32))

    def train(s, n):
        if n == 0:
            return eb.ebic_surrogate_step(s, seq, length, S, target, N, lr=1e-3, update=True)
        return eb.ebic_surrogate_train(s, n, 256, 1e-3, seq, length, S, fit, N)

    def fresh():
        s = eb.ebic_surrogate_create(h, S, 7)
        eb.ebic_surrogate_train_kernel(s, kind)
        train(s, 3)
        return s

    try:
        a, b = fresh(), fresh()
        before, grads = eb.ebic_surrogate_params(a).copy(), eb.ebic_surrogate_grads(a).copy()
        torch.cuda.synchronize()
        lost_word(a).fill_(1)
        torch.cuda.synchronize()
        with pytest.raises(eb.EbicError) as e:
            train(a, steps)
        assert e.value.status == 4                                 # EBIC_ERR_TIMEOUT
        assert_bits_equal(eb.ebic_surrogate_params(a), before, "parameters after a lost step")
        assert_bits_equal(eb.ebic_surrogate_grads(a), grads, "gradients after a lost step")
        assert int(lost_word(a)[0]) == 0                           # reported once
        for n in (steps, 0, 4):
            assert train(a, n) == train(b, n)
        assert_bits_equal(eb.ebic_surrogate_params(a), eb.ebic_surrogate_params(b), "parameters")
        eb.ebic_surrogate_free(a)
        eb.ebic_surrogate_free(b)
    finally:
        eb.ebic_free(h)


def test_lost_scores_of_a_screened_run():
    """Scores that a kernel lost end the step, or the scoring call, that finds out with
    EBIC_ERR_TIMEOUT, once; the generations stand."""
    torch = pytest.importorskip("torch")
    eb.build()
    rng = np.random.default_rng(3)
    h = eb.ebic_load_matrix(rng.standard_normal((300, C)).astype(np.float32))
    try:
        s = eb.ebic_surrogate_create(h, S, 7)
        eb.ebic_run_screen(h, s, 4, eb.SCREEN_SURROGATE)
        p = eb.ebic_default_params(pop_size=50, iterations=20, sigma=5)
        word = lost_word(s, "ebic_internal_lost_scores")
        tops = []
        for lost in (False, True):
            eb.ebic_run_init(h, p)
            eb.ebic_run_step(h, 2)
            if lost:
                word.fill_(1)
                torch.cuda.synchronize()
                with pytest.raises(eb.EbicError) as e:
                    eb.ebic_run_step(h, 3)
                assert e.value.status == 4 and int(word[0]) == 0
            else:
                eb.ebic_run_step(h, 3)
            assert eb.ebic_run_step(h, 1)["generations_done"] == 6
            tops.append(eb.ebic_get_toprank(h, 100, 6)[0])
        assert tops[0] == tops[1]
        seq = torch.zeros((5, S), dtype=torch.int16, device="cuda")
        length = torch.ones(5, dtype=torch.int32, device="cuda")
        out = torch.zeros(5, device="cuda")
        word.fill_(1)
        torch.cuda.synchronize()
        with pytest.raises(eb.EbicError) as e:
            eb.ebic_surrogate_predict(s, seq, length, S, 5, out)
        assert e.value.status == 4
        eb.ebic_surrogate_predict(s, seq, length, S, 5, out)
        eb.ebic_run_screen(h, None, 1, eb.SCREEN_OFF)
        eb.ebic_surrogate_free(s)
    finally:
        eb.ebic_free(h)
