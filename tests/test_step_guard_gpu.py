"""The FP32 walk's guard on a record that was overwritten between the count and the
emit (needs a GPU): a chunk of no candidates, which a walk that trusts it never
gets through. The emit finds it before it walks the row and reports it."""

import pytest
import torch

from paper_2401_03555_gb300 import impact, workloads as W

pytestmark = pytest.mark.gpu


ROOM, CAR = W.room_5d(cells_per_dim=9), W.unicycle_3d(nx=15, ny=13, nth=7)
FIELDS = ["chunk", "width", "magic", "table"]


# the leaf table's number is read where the emit takes lists: in the rooms
@pytest.mark.parametrize("prob,field", [(p, f) for p in (ROOM, CAR) for f in FIELDS] + [(ROOM, "leaf")],
                         ids=lambda x: x if isinstance(x, str) else x.name)
def test_an_overwritten_record_is_refused(prob, field):
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
    k = int(at[len(at) // 2])
    if field == "chunk":
        v[k + 1, 3] &= 0xffff
    elif field == "width":
        v[k, 0] = 1 << 20
    elif field == "magic":
        v[k, 3] += 1 << 24
    elif field == "table":
        v[k, 1] = 1 << 20
    else:   # behind the dimensions' entries
        v[k + 2 * prob.n, 1] = 1 << 8
    torch.cuda.synchronize()
    with pytest.raises(impact.ImpactError) as e:
        batch.emit(rb, pb, ref.nnz, ws)
    assert e.value.status == impact.IMPACT_ERR_CUDA
    assert "step guard" in str(e.value)
    again = impact.build(prob, "fp32")   # the device and the library stay usable
    assert torch.equal(again.col, ref.col) and torch.equal(again.up, ref.up)
