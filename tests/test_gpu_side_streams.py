"""Side streams are leased, not made by every worker of every call: their number
stays at the number of calls that ran at the same time, and results are the same
when leased streams pass between threads and callers' streams."""
import threading

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eod():
    import __graft_entry__ as g
    g.build()
    import paper_2506_22713_gb300 as eod
    return eod


def test_batches_do_not_grow_the_number_of_streams(eod, monkeypatch):
    monkeypatch.setenv("EOD_BATCH_STREAMS", "4")
    As = [torch.from_numpy(np.asfortranarray(W.exact_rank(m=200 + i, n=160, r=5 + i, seed=i).A)).cuda() for i in range(9)]
    before = eod.eod_abe_debug_side_streams()
    for _ in range(12):
        fs = eod.factor_batched(As, 1e-8, 3)[0]
        assert [f.rank for f in fs] == [5 + i for i in range(9)]
        for f in fs:
            f.close()
    assert eod.eod_abe_debug_side_streams() <= max(before, 4)


def test_threads_and_streams(eod):
    A = torch.from_numpy(np.asfortranarray(W.exact_rank(m=2100, n=2000, r=70, seed=2).A)).cuda()
    torch.cuda.synchronize()

    def run(stream=None):
        f = eod.factor(A, 1e-8, 3, block_k=32, stream=stream)
        out = f.rank, f.U.clone(), f.D.clone(), f.rel_err
        torch.cuda.synchronize()
        f.close()
        return out
    ref = run()
    before = eod.eod_abe_debug_side_streams()
    got = []

    def work():
        st = torch.cuda.Stream()
        for _ in range(3):
            got.append(run(st.cuda_stream))
    for _ in range(3):
        ts = [threading.Thread(target=work) for _ in range(3)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
    assert len(got) == 27
    for rank, U, D, err in got:
        assert rank == ref[0] and err == ref[3] and torch.equal(U, ref[1]) and torch.equal(D, ref[2])
    assert eod.eod_abe_debug_side_streams() <= max(before, 3)
