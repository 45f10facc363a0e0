"""What making a batch does beside filling its work list."""
import numpy as np
import pytest

import oracle
import paper_1801_03039_gb300 as eb
from helpers import assert_bits_equal, oracle_eval

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("table", [False, True])
@pytest.mark.parametrize("R,C,P", [(100, 5, 3), (9000, 30, 200)])
def test_tuning_times_only_what_it_chooses(R, C, P, table):
    """With a pair table there is nothing to choose: the problem takes it, at the
    smallest size too, and creation launches no kernel.  Without one, part sizes of
    the columns are timed."""
    import torch
    eb.build()
    oracle.build()
    rng = np.random.default_rng(R)
    A = rng.standard_normal((R, C)).astype(np.float32)
    off = np.arange(0, 3 * P + 1, 3, dtype=np.int32)
    cols = np.concatenate([rng.permutation(C)[:3] for _ in range(P)]).astype(np.int32)
    h = eb.ebic_load_matrix(A)
    try:
        if table:
            eb.ebic_build_pair_table(h)
        inc = torch.zeros(P, dtype=torch.int32, device="cuda")
        fit = torch.zeros(P, dtype=torch.float64, device="cuda")
        item = (torch.from_numpy(off).cuda(), torch.from_numpy(cols).cuda(), P, len(cols), 5, inc, fit)
        before = eb.ebic_kernel_launches()
        b = eb.ebic_batch_create([h], [item], eb.BATCH_AUTOTUNE)
        launched = eb.ebic_kernel_launches() - before
        try:
            assert (launched == 0) == table
            path = eb.ebic_batch_describe(b, 0)["path"]
            assert path == (eb.PATH_BITMASK if table else eb.PATH_GATHER)
            eb.ebic_batch_eval(b)
            torch.cuda.synchronize()
            want = oracle_eval(A, off, cols, 5)
            assert_bits_equal(inc.cpu().numpy().view(np.uint32), want[0], "inc")
            assert_bits_equal(fit.cpu().numpy(), want[2], "fitness")
        finally:
            eb.ebic_batch_free(b)
    finally:
        eb.ebic_free(h)
