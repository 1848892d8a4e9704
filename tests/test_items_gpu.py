"""Shared image tables against the oracle where they can go wrong (needs a GPU):
window widths around the lane groups and around the widest sorted window,
dimensions that read few coordinates or none, repeated inputs, windows too wide
for the tables. Tolerances are those of parity.py."""

import numpy as np
import pytest
import torch

import oracle
import parity as PA
from paper_2401_03555_gb300 import impact, workloads as W

pytestmark = pytest.mark.gpu


def linear(cells, A, sigma_cells, cutoff, inputs, B=None, seed=0):
    """x+ = A x + B u + w on [-1,1]^n with sigma in cell widths."""
    n = len(cells)
    A = np.asarray(A, np.float64)
    rng = np.random.default_rng(seed)
    U = np.asarray(inputs, np.float64)
    return W.Problem(
        name="items", kind=W.AFFINE, lo=np.full(n, -1.0), hi=np.full(n, 1.0),
        cells=np.asarray(cells, np.int32), inputs=U,
        sigma=2.0 / np.asarray(cells) * np.asarray(sigma_cells, np.float64), cutoff=cutoff, A=A,
        B=rng.normal(0.0, 0.2, (n, U.shape[1])) if B is None else np.asarray(B, np.float64),
        c=rng.uniform(-0.05, 0.05, n))


def images_of(prob, seed):
    rng = np.random.default_rng(seed)
    m = rng.uniform(-1.2, 1.2, (prob.rows, prob.n))
    return W.with_images(prob, np.stack([m, m + rng.uniform(0.0, 0.3, m.shape)], axis=2))


U1, U2 = [[-0.3], [0.4]], [[-0.3, 0.1], [0.4, 0.1], [0.4, 0.1], [0.0, -0.5]]
PROBLEMS = {
    # windows as wide as the grid: one below, at and above 8, 16 and 32 edges
    "width-7-8": lambda: linear([7, 8], np.eye(2) * 0.9, [4, 4], 1e-8, U1),
    "width-15-16": lambda: linear([15, 16], [[0.9, 0.1], [0.0, 0.8]], [6, 6], 1e-8, U1),
    "width-31-32": lambda: linear([31, 32], [[0.9, 0.0], [0.1, 0.8]], [9, 9], 1e-8, U1),
    "width-33-3": lambda: linear([33, 3], np.eye(2) * 0.9, [9, 2], 1e-8, U1),
    # the last dimension's window at and beyond the widest sorted one
    "sorted-256": lambda: linear([3, 256], np.eye(2) * 0.9, [2, 60], 1e-8, U1),
    "sorted-257": lambda: linear([3, 257], np.eye(2) * 0.9, [2, 60], 1e-8, U1),
    # windows wider than the FP64 tables (cutoff 0 keeps every cell)
    "wide-2049": lambda: linear([2049], [[0.9]], [50], 0.0, U1),
    "wide-2048": lambda: linear([2048], [[0.9]], [50], 0.0, U1),
    # a dimension that reads no coordinate, signed zeros, repeated inputs
    "no-reads": lambda: linear([6, 5, 4], [[0, 0, 0], [-0.0, 0.9, 0], [0.2, 0, 0.7]],
                               [0.8, 0.6, 0.5], 1e-8, U2),
    "crossed": lambda: linear([5, 4, 3, 4], np.roll(np.eye(4) * 0.9, 1, axis=1),
                              [0.5, 0.9, 0.4, 0.6], 1e-6, U2,
                              B=[[0.1, 0], [0, 0.1], [0, 0], [-0.0, 0]]),
    "dense-6d": lambda: linear([3, 2, 3, 2, 3, 2], np.eye(6) * 0.8 + 0.02, [0.5] * 6, 0.0, U1),
    "images": lambda: images_of(linear([9, 12], np.eye(2), [0.7, 0.5], 1e-8, U2), 3),
    # shared leaf tables around the sizes the emit pass takes by lists (20 and 48
    # entries, window bounds 64 and 160), with rows of all sizes at the border
    "lists-4x5": lambda: linear([6, 8, 8], np.eye(3) * 0.9, [0.4, 0.3, 0.4], 1e-8, U1),
    "lists-6x7": lambda: linear([5, 9, 12], np.eye(3) * 0.9, [0.5, 0.45, 0.5], 1e-8, U2),
    "lists-7x7": lambda: linear([6, 12, 12], np.eye(3) * 0.9, [0.9, 0.52, 0.5], 1e-8, U1),
    "lists-5d": lambda: linear([4, 3, 5, 9, 9], np.eye(5) * 0.9, [0.8, 0.4, 0.6, 0.45, 0.4], 1e-8, U1),
    # cutoffs around FP32's smallest normal number (pruning and searches use FP32)
    "cutoff-1e-39": lambda: linear([12, 9, 5], np.eye(3) * 0.9, [0.3, 0.4, 0.2], 1e-39, U1),
    "cutoff-1e-31": lambda: linear([12, 9, 5], np.eye(3) * 0.9, [0.3, 0.4, 0.2], 1e-31, U1),
    "cutoff-2e-30": lambda: linear([12, 9, 5], np.eye(3) * 0.9, [0.3, 0.4, 0.2], 2e-30, U1),
    "one-cell": lambda: linear([1, 1, 5], np.eye(3) * 0.5, [0.3, 1.0, 0.6], 1e-8, U1),
}


@pytest.fixture(scope="module")
def orc():
    return oracle.default()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name", list(PROBLEMS))
def test_tables_match_the_oracle(orc, name, precision):
    prob = PROBLEMS[name]()
    csr = impact.build(prob, precision)
    torch.cuda.synchronize()
    rows = np.arange(prob.rows) if prob.rows <= 2000 else W.sample_rows(prob, 200, seed=2)
    PA.compare(prob, csr, orc.build_rows(prob, rows), orc, precision).assert_ok()


def test_mixed_batch_equals_its_builds(orc):
    """Builds on and off the FP64 tables in one batch: bitwise as alone."""
    probs = [PROBLEMS[k]() for k in ("no-reads", "wide-2049", "images", "width-33-3")]
    batch = impact.Batch(probs, "fp64").build()
    for q, p in enumerate(probs):
        one, part = impact.build(p, "fp64"), batch.part(q)
        for k in ("row_ptr", "col", "lo", "up", "sink_lo", "sink_up", "trunc", "row_flags"):
            assert torch.equal(getattr(one, k), getattr(part, k)), (q, k)


# rows around one tile of the row-pointer scan (4096 rows) and around the most
# tiles that the row-terms kernels begin the scan for (152)
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("cells,inputs", [(1, 1), (64, 64), (17, 241), (64, 9728), (3, 207531)])
def test_row_pointers_at_the_scan_tiles(cells, inputs, precision):
    """Row pointers against running sums of the kept pairs of the dense build
    (exact: FP64 keeps by the same values; FP32 is checked dense)."""
    U = np.resize([[-0.3], [0.4], [0.0], [1.2]], (inputs, 1))
    dense = linear([cells], [[0.9]], [0.8], 0.0, U)
    csr = impact.build(dense, precision)
    want = torch.arange(dense.rows + 1, device="cuda") * cells
    assert torch.equal(csr.row_ptr, want)
    if precision == "fp64":
        kept = (csr.up.view(dense.rows, cells) >= 1e-3).sum(1).cumsum(0)
        got = impact.build(linear([cells], [[0.9]], [0.8], 1e-3, U), "fp64")
        assert int(got.row_ptr[0]) == 0 and torch.equal(got.row_ptr[1:], kept)
        assert got.nnz == int(kept[-1])


@pytest.mark.parametrize("cells", [[1], [2, 3], [3, 4], [5, 7], [8, 9], [2, 3, 4], [3, 2, 3, 2],
                                   [3, 2, 2, 2, 2], [2, 2, 3, 2, 2, 2], [2] * 7, [2] * 8])
def test_windows_by_lane_groups_equal_those_by_lanes(cells):
    """Few rows of distinct images make their windows by groups of lanes, rows
    beside many others by single lanes: bitwise the same. Window widths (the
    grid's, up to 9) around the group of 4; dimensions that fill a warp unevenly."""
    n = len(cells)
    A = np.eye(n) * 0.7 + 0.05
    small = linear(cells, A, [2.0] * n, 1e-9, U2)
    images = images_of(small, 5)
    big = linear([80, 80], np.eye(2) * 0.7 + 0.05, [0.6] * 2, 1e-6, U2)   # 25600 rows
    batch = impact.Batch([small, big, images], "fp32").build()
    for q, p in ((0, small), (2, images)):
        one, part = impact.build(p, "fp32"), batch.part(q)
        for k in ("row_ptr", "col", "lo", "up", "sink_lo", "sink_up", "trunc", "row_flags"):
            assert torch.equal(getattr(one, k), getattr(part, k)), (q, k)


@pytest.mark.parametrize("cells,sigma", [([12, 11, 10], 0.3), ([12, 11, 10], 0.6), ([7, 8, 9], 4.0),
                                         ([16, 17], 5.0), ([3, 31, 10], 1.1)])
def test_shared_windows_by_lane_groups_equal_those_by_lanes(cells, sigma):
    """A build of few distinct images makes its shared windows by eight lanes each, one
    of more than 12,288 by single lanes: the same inputs among many others have
    the same rows, bitwise. Widths below, at and beyond the group."""
    n, few = len(cells), 8
    many = few + 12289 // sum(cells) + 1
    U = np.random.default_rng(3).uniform(-0.5, 0.5, (many, 1))
    B = np.full((n, 1), 0.3)
    small = linear(cells, np.eye(n) * 0.9, [sigma] * n, 1e-9, U[:few], B=B)
    large = linear(cells, np.eye(n) * 0.9, [sigma] * n, 1e-9, U, B=B)
    a, b = impact.build(small, "fp32"), impact.build(large, "fp32")
    total = small.total_cells
    rows = (torch.arange(total, device="cuda")[:, None] * many
            + torch.arange(few, device="cuda")[None]).flatten()
    for k in ("sink_lo", "sink_up", "trunc", "row_flags"):
        assert torch.equal(getattr(a, k), getattr(b, k)[rows]), k
    len_a = a.row_ptr[1:] - a.row_ptr[:-1]
    assert torch.equal(len_a, b.row_ptr[rows + 1] - b.row_ptr[rows])
    at = torch.repeat_interleave(b.row_ptr[rows] - a.row_ptr[:-1], len_a) + torch.arange(
        a.nnz, device="cuda")
    for k in ("col", "lo", "up"):
        assert torch.equal(getattr(a, k), getattr(b, k)[at]), k


def repeated(count, distinct):
    return np.resize(np.random.default_rng(6).uniform(-0.4, 0.4, (distinct, 1)), (count, 1))


# input lists around the longest whose classes are all found, with few and many
# distinct points; caller images whose windows are far narrower than the grid, of
# different widths side by side
MORE = {
    "inputs-2048": lambda: linear([5, 4], np.eye(2) * 0.9, [0.6, 0.5], 1e-8, repeated(2048, 2048)),
    "inputs-2049": lambda: linear([5, 4], np.eye(2) * 0.9, [0.6, 0.5], 1e-8, repeated(2049, 2049)),
    "inputs-cycle": lambda: linear([5, 4, 3], np.eye(3) * 0.9, [0.6, 0.5, 0.4], 1e-8, repeated(5001, 7)),
    "inputs-long-cycle": lambda: linear([5, 4, 3], np.eye(3) * 0.9, [0.6, 0.5, 0.4], 1e-8,
                                        repeated(9000, 4500)),
    "images-70": lambda: images_of(linear([70], np.eye(1), [1.0], 1e-8, U2), 3),
    "images-40x300": lambda: images_of(linear([40, 300], np.eye(2), [0.6, 5.0], 1e-8, U1), 4),
    "images-outside": lambda: images_of(linear([33, 35], np.eye(2), [0.02, 0.02], 1e-3, U1), 5),
}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name", list(MORE))
def test_long_input_lists_and_narrow_windows_match_the_oracle(orc, name, precision):
    prob = MORE[name]()
    csr = impact.build(prob, precision)
    torch.cuda.synchronize()
    rows = np.arange(prob.rows) if prob.rows <= 2000 else W.sample_rows(prob, 200, seed=2)
    PA.compare(prob, csr, orc.build_rows(prob, rows), orc, precision).assert_ok()
