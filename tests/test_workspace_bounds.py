"""Scratch that a build asks of its caller (host-only sizing, no GPU): tables that
only save time stay within fixed bounds on grids whose images are all distinct."""

import numpy as np
import pytest

from paper_2401_03555_gb300 import impact, workloads as W


def distinct(n, cells, inputs, kind):
    """Every row its own image: dense dynamics, or images the caller brings."""
    return W.Problem(name="distinct", kind=kind, lo=np.full(n, -1.0), hi=np.full(n, 1.0),
                     cells=np.full(n, cells, np.int32),
                     inputs=np.linspace(-0.5, 0.5, inputs)[:, None],
                     sigma=np.full(n, 2.0 / cells), cutoff=1e-8, A=0.9 * np.eye(n) + 0.01,
                     B=np.full((n, 1), 0.2), c=np.zeros(n))


@pytest.mark.parametrize("kind", [W.AFFINE, W.IMAGES])
@pytest.mark.parametrize("n,cells,inputs", [(2, 40, 27), (2, 100, 27), (3, 50, 27), (3, 100, 27),
                                            (4, 30, 9), (4, 30, 27), (2, 1000, 4)])
def test_fp64_workspace_is_bounded(kind, n, cells, inputs):
    prob = distinct(n, cells, inputs, kind)
    # the item tables, 24 bytes a row, the descriptor and its tables
    assert impact.workspace_bytes(prob, "fp64") <= (1 << 30) + 24 * prob.rows + (64 << 20)
