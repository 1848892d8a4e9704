"""Synthesis over cell counts at which the values are ranked in other ways (needs a
GPU): counted up to 4096 cells, sorted by tiles of 2048 and merge passes beyond,
ranks of 16 bits up to 65533 cells. A disjoint union of small IMDPs has each
one's own values, bitwise: no rank compares across more than its order."""

from dataclasses import replace
from functools import lru_cache
from types import SimpleNamespace

import numpy as np
import pytest
import torch

from paper_2401_03555_gb300 import impact, workloads as W

pytestmark = pytest.mark.gpu

PARTS, SIDE = 11, 9
CELLS = SIDE * SIDE
INPUTS = 9


@lru_cache(maxsize=None)
def part(k, precision):
    """One of a few robots of 81 cells: its IMDP and labels (target, avoid)."""
    rng = np.random.default_rng(100 + k)
    prob = replace(W.robot_2d(cells_per_dim=SIDE), c=rng.uniform(-0.4, 0.4, 2),
                   sigma=rng.uniform(0.6, 1.2, 2))
    lo = rng.uniform(-9.0, 3.0, 2)
    labels = impact.label_cells(prob, target=[(lo, lo + 5.0)], avoid=[(-lo - 2.0, -lo + 1.5)])
    return impact.build(prob, precision), labels


def union(cells, kinds, precision):
    """As many parts as fit into `cells` cells, in turn, and labelled cells (their
    rows empty, never used) at the end."""
    parts = [part(k % kinds, precision) for k in range(cells // CELLS)]
    pad = cells - len(parts) * CELLS
    one = torch.cat([p[0].row_ptr[1:] - p[0].row_ptr[:-1] for p in parts]
                    + [torch.zeros(pad * INPUTS, dtype=torch.int64, device="cuda")])
    row_ptr = torch.zeros(cells * INPUTS + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(one, 0, out=row_ptr[1:])

    def rows(name, fill):
        t = [getattr(p[0], name) for p in parts]
        return torch.cat(t + [torch.full((pad * INPUTS,), fill, dtype=t[0].dtype, device="cuda")])

    csr = impact.CSR(precision, row_ptr,
                     torch.cat([p[0].col + k * CELLS for k, p in enumerate(parts)]).int(),
                     torch.cat([p[0].lo for p in parts]), torch.cat([p[0].up for p in parts]),
                     rows("sink_lo", 0.0), rows("sink_up", 1.0), rows("trunc", 0.0),
                     rows("row_flags", 0))
    labels = torch.cat([p[1] for p in parts]
                       + [1 + torch.arange(pad, device="cuda", dtype=torch.uint8) % 2])
    return csr, labels.to(torch.uint8)


def run(csr, labels, **kw):
    prob = SimpleNamespace(total_cells=labels.numel(), n_inputs=INPUTS)
    return impact.synthesize(csr, prob, labels, **kw)


def check(cells, kinds, precision, **kw):
    got = run(*union(cells, kinds, precision), **kw)
    alone = [run(*part(k, precision), **kw) for k in range(kinds)]
    for f in ("p_min", "p_max", "policy"):
        n = cells // CELLS
        want = torch.cat([getattr(alone[k % kinds], f) for k in range(n)])
        assert torch.equal(getattr(got, f)[:n * CELLS], want), f
    return got, alone


# one tile beyond the counted ranks and cells that fill, miss and just start
# tiles: even, odd and many runs to merge; the last of the 16-bit ranks
SIZES = [4095, 4096, 4097, 6144, 6145, 10243, 18433, 65533, 65534, 70001]


@pytest.mark.parametrize("cells", SIZES)
@pytest.mark.parametrize("spec,optimistic", [(impact.REACH_AVOID, False), (impact.SAFETY, False),
                                             (impact.REACH_AVOID, True)])
def test_a_union_of_parts_has_each_ones_values(cells, spec, optimistic):
    precision = "fp32" if cells % 2 else "fp64"
    check(cells, PARTS, precision, spec=spec, optimistic=optimistic, horizon=12)


@pytest.mark.parametrize("cells", [4097, 6145, 65534])
@pytest.mark.parametrize("max_iters", [1, 7, 8, 9, 10000])
def test_the_stopping_test_on_the_device(cells, max_iters):
    """Equal parts stop together: the iterations of one alone, at a limit below, at
    and beyond the launches that go out together, and where the bounds meet."""
    eps = 1e-4 if max_iters == 10000 else 1e-14
    got, alone = check(cells, 1, "fp64", eps=eps, max_iters=max_iters)
    assert got.iterations == alone[0].iterations
    assert max(got.iterations) == max_iters or max_iters == 10000
    assert max(got.iterations) < 10000
