"""Builds from several host threads at once (needs a GPU): every entry point may
be called from several threads, so builds of different sizes beside each other
finish with the bits they have alone."""

import threading
from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2401_03555_gb300 import impact, workloads as W

pytestmark = pytest.mark.gpu

FIELDS = ("row_ptr", "col", "lo", "up", "sink_lo", "sink_up", "trunc", "row_flags")


# launches of little and of much shared memory: narrow windows, many
# dimensions, wide windows
PROBLEMS = [lambda: W.robot_2d(cells_per_dim=7), lambda: W.room_5d(cells_per_dim=5),
            lambda: replace(W.robot_2d(cells_per_dim=60), sigma=np.array([5.0, 5.0]), cutoff=1e-8)]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_builds_of_different_sizes_run_beside_each_other(precision):
    problems = [make() for make in PROBLEMS]
    alone = [impact.build(p, precision) for p in problems]
    torch.cuda.synchronize()
    failed = []

    def work(p, ref):
        try:
            b = impact.Builder(p, precision, capacity=ref.nnz)
            s = torch.cuda.Stream()
            for _ in range(400):
                b.run(stream=s)
            got = b.result()
            for f in FIELDS:
                assert torch.equal(getattr(got, f), getattr(ref, f)), f
        except Exception as e:   # reported by the test's own thread
            failed.append((p.name, repr(e)))

    threads = [threading.Thread(target=work, args=a) for a in zip(problems, alone) for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
