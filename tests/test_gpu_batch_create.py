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


def test_work_of_every_length():
    """Series of every length from 1 to 40 and of 1,024, invalid ones among them, in
    problems of one part and of several: each item is taken once, whatever its
    place in the list."""
    import torch
    eb.build()
    oracle.build()
    rng = np.random.default_rng(3)
    handles, items, want, outs = [], [], [], []
    try:
        for R, C, P in ((50, 60, 90), (30000, 41, 300), (700, 50, 1)):
            A = rng.standard_normal((R, C)).astype(np.float32)
            lens = [int(v) for v in rng.integers(1, 41, P)]
            lens[-1] = 1024
            seqs = [np.sort(rng.permutation(C)[:n]) if n <= C else rng.integers(0, C, n) for n in lens]
            off = np.cumsum([0] + lens).astype(np.int32)
            cols = np.concatenate(seqs).astype(np.int32)
            inc, _, fit = oracle_eval(A, off, cols, 4)
            if P > 1:
                off = np.concatenate([off, [off[-1], off[-1] + 1100]]).astype(np.int32)   # 0, 1,100
                cols = np.concatenate([cols, np.zeros(1100, np.int32)])
                inc, fit = np.append(inc, [0, 0]).astype(np.uint32), np.append(fit, [0.0, 0.0])
            h = eb.ebic_load_matrix(A)
            handles.append(h)
            if R != 700:
                eb.ebic_build_pair_table(h)
            n = len(off) - 1
            o = (torch.full((n,), -1, dtype=torch.int32, device="cuda"),
                 torch.full((n,), -1.0, dtype=torch.float64, device="cuda"))
            outs.append(o)
            want.append((inc, fit))
            items.append((torch.from_numpy(off).cuda(), torch.from_numpy(cols).cuda(), n, len(cols), 4) + o)
        b = eb.ebic_batch_create(handles, items, 0)
        try:
            d = [eb.ebic_batch_describe(b, k) for k in range(3)]
            assert d[1]["parts"] > 1
            assert d[0]["work_items"] == sum(x["parts"] * it[2] for x, it in zip(d, items))
            eb.ebic_batch_eval(b)
            torch.cuda.synchronize()
        finally:
            eb.ebic_batch_free(b)
        for (inc, fit), (wi, wf) in zip(outs, want):
            assert_bits_equal(inc.cpu().numpy().view(np.uint32), wi, "inc")
            assert_bits_equal(fit.cpu().numpy(), wf, "fitness")
    finally:
        for h in handles:
            eb.ebic_free(h)
