"""GPU: handles of several host threads at once, whose products launch the same
kernels with different amounts of shared memory."""
import threading

import numpy as np
import pytest

from paper_2103_11991_gb300 import inputs as I
from tests._gpu import check_against_oracle

pytestmark = pytest.mark.gpu


def test_threads_with_rows_of_different_sizes():
    import torch
    from paper_2103_11991_gb300 import spgemm as K
    # rank rows of 250 and of 1,000 columns, unsorted ones, wide rows of narrow and of wide B
    wide = {"force_tier": 2, "structure_cache": 0}
    shapes = [(30000, 15, 17, {}), (60000, 31, 33, {}), (9000, 20, 30, {"unsorted": True}),
              (60000, 20, 30, {"unsorted": True}), (5000, 60, 70, wide), (200000, 60, 70, wide),
              (100000, 60, 70, wide), (300000, 60, 70, wide)]
    jobs, errors = [], []
    for n, lo, hi, o in shapes:
        A = I.random_rows(300, 500, lo, hi, seed=n, purpose="thA")
        B = I.random_rows(500, n, lo, hi, seed=n + 1, purpose="thB")
        if o.get("unsorted"):
            B.colind = np.concatenate([B.colind[B.rowptr[i]:B.rowptr[i + 1]][::-1] for i in range(B.m)])
        opts = {k: v for k, v in o.items() if k != "unsorted"}
        jobs.append((A, B, K.DeviceCSR.from_host(A), K.DeviceCSR.from_host(B), opts))
    torch.cuda.synchronize()
    start = threading.Barrier(len(jobs))
    results = [None] * len(jobs)

    def work(t):
        A, B, dA, dB, opts = jobs[t]
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream), K.SpGEMM(stream=stream, arith=1, small_max_rows=0, **opts) as op:
                start.wait(60)
                rp, nnz = op.symbolic(dA, dB)
                ci, va = op.numeric(dA, dB, rp, nnz)
                for _ in range(300):
                    op.symbolic(dA, dB)
                    for _ in range(5):
                        op.numeric(dA, dB, rp, nnz, ci, va)
                op.sync()
                results[t] = tuple(x.cpu().numpy() for x in (rp, ci, va))
        except Exception as e:  # noqa: BLE001
            errors.append((t, repr(e)))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for (A, B, *_), got in zip(jobs, results):
        check_against_oracle(A, B, *got)
