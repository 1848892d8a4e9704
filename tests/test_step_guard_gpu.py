"""The FP32 walk's guard on a record that was overwritten between the count and the
emit (needs a GPU): a chunk of no candidates, which a walk that trusts it never
gets through. The emit finds it before it walks the row and reports it."""

import pytest
import torch

from paper_2401_03555_gb300 import impact, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prob", [W.room_5d(cells_per_dim=5), W.unicycle_3d(nx=15, ny=13, nth=7)],
                         ids=lambda p: p.name)
def test_a_chunk_of_no_candidates_ends_the_walk(prob):
    ref = impact.build(prob, "fp32")
    batch = impact.Batch([prob], "fp32")
    rb, pb = impact.alloc_rows(prob.rows), impact.alloc_pairs(ref.nnz, "fp32")
    ws = batch.alloc_workspace()
    assert batch.count(rb, ws) == ref.nnz
    torch.cuda.synchronize()
    # the entries of dimension 0 in the rows' records, 16-byte aligned: width tw
    # first, column stride and lay = 32 / tw parents | (64 / tw) tw << 16 last
    v = ws[:ws.numel() // 16 * 16].view(torch.int32).view(-1, 4)
    a, b = v[:-1], v[1:]
    tw = a[:, 0].clamp(1, 32)
    stride = int(prob.total_cells // int(prob.cells[0]))
    hit = ((a[:, 0] == tw) & (b[:, 2] == stride)
           & (b[:, 3] == torch.div(32, tw, rounding_mode="floor")
              + ((torch.div(64, tw, rounding_mode="floor") * tw) << 16)))
    at = torch.nonzero(hit).flatten()
    assert len(at) >= prob.rows // 2
    k = int(at[len(at) // 2]) + 1
    v[k, 3] &= 0xffff
    torch.cuda.synchronize()
    with pytest.raises(impact.ImpactError) as e:
        batch.emit(rb, pb, ref.nnz, ws)
    assert e.value.status == impact.IMPACT_ERR_CUDA
    assert "step guard" in str(e.value)
    again = impact.build(prob, "fp32")   # the device and the library stay usable
    assert torch.equal(again.col, ref.col) and torch.equal(again.up, ref.up)
