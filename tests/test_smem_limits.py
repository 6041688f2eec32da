"""A kernel's limit of dynamic shared memory belongs to the kernel, not to one
launch of it: it is set in one place, always to the same value, so that a
thread that launches a kernel with little does not refuse another's launch
with much."""
from __future__ import annotations

import glob
import os
import re
import threading

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2106_13062_gb300", "csrc")


def test_one_place_sets_the_limit():
    calls = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for m in re.finditer(r"cudaFuncSetAttribute\([^;\"]+,\s*cudaFuncAttribute", open(path).read()):
            calls.append((os.path.basename(path), m.start()))
    assert [c[0] for c in calls] == ["fcs_internal.cuh"], calls


@pytest.mark.gpu
@pytest.mark.parametrize("last", [256, 255])
def test_two_threads_two_sizes(last):
    """One kernel from two threads with two contexts, with much and with
    little shared memory (256: the row kernel, 255: the general one)."""
    import torch

    import paper_2106_13062_gb300 as fcs
    fcs.build()
    failed = []

    def work(J):
        with torch.cuda.stream(torch.cuda.Stream()):
            ctx = fcs.Context()
            I = [8, 8, last]
            h, s = fcs.fcs_make_hashes(ctx, 3, I, J, 10)
            T = torch.zeros(*I, device="cuda")
            out = None
            for k in range(6000):
                try:
                    out = fcs.fcs_sketch_dense(ctx, T, J, h, s, out=out)
                except fcs.FcsError as e:
                    failed.append(str(e))
                    break
                if k % 64 == 0:
                    torch.cuda.current_stream().synchronize()
            torch.cuda.current_stream().synchronize()
            ctx.close()

    threads = [threading.Thread(target=work, args=([j] * 3,)) for j in (1500, 500)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not failed, failed
