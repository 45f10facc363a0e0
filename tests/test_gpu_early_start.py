"""Evaluation kernels come up while the kernel before them in the stream runs.
What that kernel writes -- the population itself, or the results and counters of
another evaluation -- must be complete before they touch it."""
import numpy as np
import pytest

import oracle
import paper_1801_03039_gb300 as eb
from helpers import assert_bits_equal, oracle_eval

pytestmark = pytest.mark.gpu

# (rows, table, launch shape): lane, warp (whole and split), staged and phased
# kernels over the table; rank planes of one slice and of several, fp32 columns
SHAPES = [(1500, True, dict(kernel=1)), (1500, True, dict(kernel=2)),
          (9000, True, dict(kernel=2, vecs_per_part_bitmask=32)),
          (9000, True, dict(kernel=3, dense_steps=2)), (9000, True, dict(kernel=4, dense_steps=2)),
          (900, False, {}), (9000, False, {}), (9000, False, dict(vecs_per_part_gather=64))]


@pytest.mark.parametrize("both", [False, True])
@pytest.mark.parametrize("R,table,shape", SHAPES)
def test_population_written_right_before(R, table, shape, both):
    """Forty evaluations queued without a wait, each of a population that a copy
    kernel has just written over the one before, into the same outputs, which a copy
    kernel takes away right after; and pairs of evaluations into the same outputs."""
    import torch
    eb.build()
    oracle.build()
    rng = np.random.default_rng(R)
    C, P, N = 25, 200, 40
    A = rng.standard_normal((R, C)).astype(np.float32)
    lens = rng.permutation(np.repeat([2, 3, 4, 5], P // 4))
    off = np.cumsum([0] + [int(n) for n in lens]).astype(np.int32)
    pops = [np.concatenate([rng.permutation(C)[:n] for n in lens]).astype(np.int32) for _ in range(4)]
    mode = 1 if both else 0
    want = [oracle_eval(A, off, p, 7, mode) for p in pops]
    h = eb.ebic_load_matrix(A)
    try:
        if table:
            eb.ebic_build_pair_table(h)
            torch.cuda.synchronize()
        eb.ebic_set_path(h, eb.PATH_BITMASK if table else eb.PATH_GATHER)
        eb.ebic_set_eval_tuning(h, **shape)
        src = [torch.from_numpy(p).cuda() for p in pops]
        d_off0 = torch.from_numpy(off).cuda()
        d_off, d_cols = torch.zeros_like(d_off0), torch.zeros_like(src[0])
        inc = torch.zeros(P, dtype=torch.int32, device="cuda")
        dec = torch.zeros_like(inc) if both else None
        fit = torch.zeros(P, dtype=torch.float64, device="cuda")
        took = [(torch.zeros_like(inc), torch.zeros_like(inc), torch.zeros_like(fit)) for _ in range(N)]
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            for k in range(N):
                d_off.zero_()
                d_cols.copy_(src[k % 4])
                d_off.copy_(d_off0)
                for _ in range(1 + k % 2):
                    eb.ebic_eval_population_dev(h, d_off, d_cols, P, len(pops[0]), 7, mode, inc, dec,
                                                fit, stream)
                took[k][0].copy_(inc)
                if both:
                    took[k][1].copy_(dec)
                took[k][2].copy_(fit)
        stream.synchronize()
        eb.ebic_check_device_error(h)
        for k in range(N):
            assert_bits_equal(took[k][0].cpu().numpy().view(np.uint32), want[k % 4][0], ("inc", k))
            if both:
                assert_bits_equal(took[k][1].cpu().numpy().view(np.uint32), want[k % 4][1], ("dec", k))
            assert_bits_equal(took[k][2].cpu().numpy(), want[k % 4][2], ("fitness", k))
    finally:
        torch.cuda.synchronize()
        eb.ebic_free(h)
