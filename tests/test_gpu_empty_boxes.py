"""Ghost boxes of no cells (lo == hi, or hi < lo, along some axis) among the
boxes of a level's ghost fill are no-ops: the fill gives what it gives without
them.  One of them lies where the parent has no cells."""
import ctypes

import numpy as np
import pytest

import paper_1307_2265_gb300 as ez
from gpu_helpers import batch_from_patches, white_patch
from paper_1307_2265_gb300 import hierarchy as gh

pytestmark = pytest.mark.gpu
EMPTY = [((5, 5, 5), (5, 9, 9)), ((5, 5, 5), (9, 5, 5)), ((5, 7, 5), (9, 9, 5)), ((7, 5, 5), (6, 9, 9)),
         ((4001, 4001, 4001), (4001, 4001, 4001))]


def _links(rows):
    import torch
    return torch.tensor(rows, dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("precision", [ez.FP64, ez.FP32])
def test_empty_interpolation_boxes_are_no_ops(precision):
    import torch
    old = batch_from_patches([white_patch((8, 8, 8), seed=1)], [0.1] * 3)
    new = batch_from_patches([white_patch((8, 8, 8), seed=2)], [0.1] * 3)
    n, origin = [(6, 8, 6)], [(4, 4, 6)]
    boxes = gh.interp_boxes_general(n, origin)
    extra = np.zeros(len(EMPTY), dtype=boxes.dtype)
    for i, (lo, hi) in enumerate(EMPTY):
        extra["lo"][i], extra["hi"][i] = lo, hi
    mixed = np.concatenate([extra[:2], boxes[:5], extra[2:], boxes[5:]])
    flinks, plinks = _links([[*origin[0], 0]]), _links([[0, 0, 0, -1]])
    pold = (ctypes.c_void_p * 5)(*[u.data_ptr() for u in old.U])
    out = []
    for table in (boxes, mixed):
        fine = batch_from_patches([white_patch(n[0], seed=3)], [0.05] * 3)
        dev = torch.from_numpy(table.view(np.uint8).copy()).cuda()
        f, p = fine.c(), new.c()
        rc = gh._lib().enzo_ghost_fill_level(ctypes.byref(f), flinks.data_ptr(), ctypes.byref(p), plinks.data_ptr(),
                                             pold, None, 0.25, dev.data_ptr(), len(table), None, 0, precision, 2)
        assert rc == 0
        torch.cuda.synchronize()
        out.append([u.cpu().numpy() for u in fine.U])
    before = white_patch(n[0], seed=3)
    for a, b, c in zip(out[0], out[1], before):
        assert np.array_equal(a, b)
        assert not np.array_equal(a, c.ravel())
