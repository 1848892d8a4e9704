"""Sampled noise by draw masks against the oracle (needs a GPU): draw counts
around the 32-draw words and the words per lane, one dimension and several,
draws that leave the domain, a single draw as the least count kept. Counts are
whole numbers: every value must be equal."""

import numpy as np
import pytest

import oracle
from paper_2401_03555_gb300 import impact, workloads as W

pytestmark = pytest.mark.gpu


def prob_of(cells, cutoff):
    n = len(cells)
    return W.Problem(name="mc-masks", kind=W.AFFINE, lo=np.full(n, -1.0), hi=np.full(n, 1.0),
                     cells=np.asarray(cells, np.int32),
                     inputs=np.array([[-0.4], [0.0], [0.0], [0.7]]), sigma=np.full(n, 0.1),
                     cutoff=cutoff, A=0.9 * np.eye(n), B=np.ones((n, 1)), c=np.full(n, 0.01))


CASES = [([9], 1), ([9, 7], 31), ([5, 4, 6], 32), ([64], 33), ([7, 5], 1023), ([4, 3, 5], 1024),
         ([6, 6], 1025), ([3, 3, 3, 3], 2048), ([8, 5], 2049), ([5, 6], 4096), ([5, 6], 4097)]


@pytest.mark.parametrize("cells,draws", CASES)
def test_masks_equal_the_oracle(cells, draws):
    w = np.random.default_rng(draws).normal(size=(draws, len(cells))) * 0.4
    for cutoff in (0.5 / draws, 2.5 / draws + 1e-3):   # one draw keeps a target; a few do
        prob = prob_of(cells, min(cutoff, 0.9))
        got = impact.build_mc(prob, w, "fp64")
        rows = np.arange(prob.rows)
        ref = oracle.build_rows_mc(prob, w, rows)
        rp = got.row_ptr.cpu().numpy()
        col, lo, up = got.col.cpu().numpy(), got.lo.cpu().numpy(), got.up.cpu().numpy()
        for r in rows:
            a, b = rp[r], rp[r + 1]
            rc, rlo, rup = ref.row(r)
            assert np.array_equal(col[a:b], rc), (cutoff, r)
            assert np.array_equal(lo[a:b], rlo) and np.array_equal(up[a:b], rup), (cutoff, r)
        for g, x in ((got.sink_lo, ref.sink_lo), (got.sink_up, ref.sink_up), (got.trunc, ref.trunc)):
            assert np.array_equal(g.cpu().numpy(), x)


def test_more_than_64_window_cells_are_refused():
    w = np.random.default_rng(0).normal(size=(100, 1)) * 50.0
    with pytest.raises(impact.ImpactError) as e:
        impact.build_mc(prob_of([65], 1e-2), w)
    assert e.value.status == impact.IMPACT_ERR_ARG
