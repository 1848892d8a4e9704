"""Builds that go without the tables that only save time (needs a GPU): when the
scratch with them cannot be had, the call runs with less and makes the same
pairs. The allocation failures are made on the host."""

import numpy as np
import pytest
import torch

import oracle
import parity as PA
from paper_2401_03555_gb300 import impact, workloads as W

pytestmark = pytest.mark.gpu


def dense_2d(cells=40, inputs=27):
    """43,200 rows, each with images of its own: 50 MB of FP64 item tables."""
    return W.Problem(name="dense2d", kind=W.AFFINE, lo=np.full(2, -1.0), hi=np.full(2, 1.0),
                     cells=np.full(2, cells, np.int32),
                     inputs=np.linspace(-0.5, 0.5, inputs)[:, None], sigma=np.full(2, 2.0 / cells),
                     cutoff=1e-8, A=np.array([[0.9, 0.05], [-0.03, 0.8]]), B=np.full((2, 1), 0.2),
                     c=np.zeros(2))


# FP64 items, FP32 leaf tables (also by the emit's lists in the rooms)
LARGE = {"fp64": [dense_2d], "fp32": [lambda: W.unicycle_3d(nx=31, ny=31, nth=17),
                                      lambda: W.room_5d(cells_per_dim=9)]}
CASES = [(p, make) for p, makes in LARGE.items() for make in makes]


def without_tables(call):
    """Runs `call` with its first allocation, the scratch, failing once."""
    impact.fail_alloc(1)
    try:
        return call()
    finally:
        impact.fail_alloc(0)


def assert_same(got, ref, precision, targets):
    for f in ("row_ptr", "col", "lo", "up", "sink_lo", "sink_up", "row_flags"):
        assert torch.equal(getattr(got, f), getattr(ref, f)), f
    if precision == "fp32":
        assert torch.equal(got.trunc, ref.trunc)
    else:   # sums of at most `targets` terms that add up to at most 1, in two orders
        assert float((got.trunc - ref.trunc).abs().max()) <= 2 * targets * 2.0 ** -53


@pytest.mark.parametrize("precision,make", CASES)
def test_builds_without_tables_make_the_same_pairs(precision, make):
    prob = make()
    ref = impact.build(prob, precision)
    batch = impact.Batch([prob], precision)
    rb, pb = impact.alloc_rows(prob.rows), impact.alloc_pairs(ref.nnz, precision)
    base = impact.live_bytes()

    def result():
        torch.cuda.synchronize()
        return impact.CSR(precision, rb["row_ptr"], pb["col"], pb["lo"], pb["up"], rb["sink_lo"],
                          rb["sink_up"], rb["trunc"], rb["row_flags"])

    def clear():
        for t in list(rb.values()) + list(pb.values()):
            t.fill_(-3)

    assert without_tables(lambda: batch.count(rb)) == ref.nnz
    without_tables(lambda: batch.emit(rb, pb, ref.nnz))
    assert_same(result(), ref, precision, prob.total_cells)
    clear()
    assert without_tables(lambda: batch.build_into(rb, pb, ref.nnz)) == ref.nnz
    assert_same(result(), ref, precision, prob.total_cells)
    clear()
    graph = without_tables(lambda: batch.graph(rb, pb, ref.nnz))
    graph.launch()
    torch.cuda.synchronize()
    assert graph.result() == ref.nnz
    assert_same(result(), ref, precision, prob.total_cells)
    graph.close()
    assert impact.live_bytes() == base


def test_one_pass_scratch_holds_no_leaf_tables():
    """The one-pass walk reads none: its own scratch is smaller than the two-pass
    build's by the leaf tables (16 MB of them or more), and the pairs are the same."""
    prob = W.unicycle_3d(nx=31, ny=31, nth=17)
    ref = impact.build(prob, "fp32")
    rb, pb = impact.alloc_rows(prob.rows), impact.alloc_pairs(ref.nnz, "fp32")
    base = impact.live_bytes()[0]
    held = []
    for one_pass in (False, True):
        batch = impact.Batch([prob], "fp32", tune=impact.tuning(one_pass=one_pass))
        graph = batch.graph(rb, pb, ref.nnz)
        held.append(impact.live_bytes()[0] - base)
        graph.launch()
        torch.cuda.synchronize()
        assert graph.result() == ref.nnz
        graph.close()
        assert torch.equal(pb["col"], ref.col) and torch.equal(pb["up"], ref.up)
        pb["col"].fill_(-3)
        assert batch.build_into(rb, pb, ref.nnz) == ref.nnz
        assert torch.equal(pb["col"], ref.col) and torch.equal(rb["trunc"], ref.trunc)
    assert held[1] <= held[0] - (16 << 20)


def test_build_without_the_callers_scratch(monkeypatch):
    """impact.build when torch cannot give the workspace: the library's own."""
    prob = dense_2d()
    ref = impact.build(prob, "fp64")
    empty = torch.empty

    def short(*size, **kw):
        if kw.get("dtype") is torch.uint8:
            raise torch.OutOfMemoryError("no workspace")
        return empty(*size, **kw)
    monkeypatch.setattr(torch, "empty", short)
    got = impact.build(prob, "fp64")
    monkeypatch.undo()
    assert_same(got, ref, "fp64", prob.total_cells)


def test_a_request_that_fits_the_budget_without_tables_is_served():
    prob = dense_2d()
    ref = impact.build(prob, "fp64")
    small = W.robot_2d(cells_per_dim=7)
    ref_small = impact.build(small, "fp64")
    assert impact.workspace_bytes(prob, "fp64") > 32 << 20
    with impact.Server("fp64", memory_budget=32 << 20, max_batch=4) as srv:
        tickets = [srv.submit(p) for p in (small, prob)]
        for t, r, p in zip(tickets, (ref_small, ref), (small, prob)):
            srv.poll(t, wait=True)
            assert_same(srv.result(t), r, "fp64", p.total_cells)
            srv.release(t)


def test_images_beyond_the_item_tables_match_the_oracle():
    """270,000 rows of caller images whose windows span the grid would take 2 GB
    of FP64 items: built pair by pair, without."""
    base = dense_2d(cells=100)
    rng = np.random.default_rng(4)
    m = rng.uniform(-1.1, 1.1, (base.rows, 2))
    prob = W.with_images(base, np.stack([m, m + rng.uniform(0.0, 0.05, m.shape)], axis=2))
    assert impact.workspace_bytes(prob, "fp64") < 64 << 20
    csr = impact.build(prob, "fp64")
    torch.cuda.synchronize()
    orc = oracle.default()
    rows = W.sample_rows(prob, 200, seed=2)
    PA.compare(prob, csr, orc.build_rows(prob, rows), orc, "fp64").assert_ok()


@pytest.mark.parametrize("mode", ["box", "cells"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_region_vectors_without_tables_have_the_same_bits(mode, precision):
    """200 x 200 x 2 cells, 4 inputs: 320,000 images of two coordinates, whose
    factors of the domain and 3 boxes take 20 MB."""
    prob = W.Problem(name="regions", kind=W.AFFINE, lo=np.full(3, -1.0), hi=np.full(3, 1.0),
                     cells=np.array([200, 200, 2], np.int32),
                     inputs=np.linspace(-0.5, 0.5, 4)[:, None], sigma=np.array([0.02, 0.02, 0.5]),
                     cutoff=1e-8, A=np.array([[0.9, 0.05, 0], [-0.03, 0.8, 0], [0, 0, 0.7]]),
                     B=np.array([[0.2], [0.1], [0.3]]), c=np.zeros(3))

    def vectors(boxes):
        r = impact.region_vectors(prob, target=boxes[:1], avoid=boxes[1:], mode=mode,
                                  precision=precision)
        return [r.r_lo, r.r_up, r.a_lo, r.a_up]

    boxes = [([-1.0 + 0.4 * i, -0.9, -1.0], [-0.8 + 0.4 * i, 0.3, 1.0]) for i in range(3)]
    ref = vectors(boxes)
    assert all(torch.equal(a, b) for a, b in zip(without_tables(lambda: vectors(boxes)), ref))


# room for the kept entries refused (286 MB): every row is walked again; the masks
# refused (25 MB, fewer entries): the per-row histograms
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("name,draws", [("room", 300), ("cube", 2100)])
def test_sampled_noise_without_its_scratch_has_the_same_bits(name, draws, precision):
    if name == "room":
        prob = W.room_5d(cells_per_dim=6)
    else:
        prob = W.Problem(name="cube", kind=W.AFFINE, lo=np.full(4, -1.0), hi=np.full(4, 1.0),
                         cells=np.array([8, 8, 8, 7], np.int32), inputs=np.zeros((1, 1)),
                         sigma=np.full(4, 0.1), cutoff=1e-3, A=0.9 * np.eye(4) + 0.05 *
                         (np.ones((4, 4)) - np.eye(4) - np.roll(np.eye(4), 1, axis=1)),
                         B=np.zeros((4, 1)), c=np.zeros(4))
    w = np.random.default_rng(draws).normal(size=(draws, prob.n)) * np.asarray(prob.sigma)
    ref = impact.build_mc(prob, w, precision, cutoff=4e-3)
    impact.fail_alloc(6)   # the five row arrays, then the scratch
    try:
        got = impact.build_mc(prob, w, precision, cutoff=4e-3)
    finally:
        impact.fail_alloc(0)
    assert ref.nnz > prob.rows
    for f in ("row_ptr", "col", "lo", "up", "sink_lo", "sink_up", "trunc", "row_flags"):
        assert torch.equal(getattr(got, f), getattr(ref, f)), f
