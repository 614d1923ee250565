"""Box types of a tree whose lists of a level end at entry 2^32 - 1, the largest that
row starts hold: the entries of a small tree, at the end of an array of that length,
give the types that they give at its start."""
import ctypes as C

import numpy as np
import pytest

from paper_1301_1704_gb300 import fmmds, workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("lists", ["e4", "e2"])
@pytest.mark.parametrize("lpar", [2, 3])
def test_rows_that_end_at_the_largest_offset(lists, lpar):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1301_1704_gb300 import build
    build.build()
    ctx = fmmds.Context(0)
    pts = torch.from_numpy(workloads.uniform(6000, 51)).cuda()
    tree = ctx.build(pts, pts, L=4)
    owner = torch.from_numpy(np.random.default_rng(lpar).integers(
        0, 3, size=tree.src.nbox[lpar]).astype(np.int32)).cuda()
    want = ctx.box_types(tree, lpar, owner, 1)
    rows, entries = getattr(tree, lists + "_off"), getattr(tree, lists + "_idx")
    kept = []
    entries_at_end = torch.zeros(2 ** 32 - 1, dtype=torch.int32, device="cuda")
    for l in (2, 3, 4):  # one level at a time: the array is 17 GB
        n = entries[l].numel()
        first = 2 ** 32 - 1 - n
        entries_at_end.zero_()
        entries_at_end[first:] = entries[l]
        far = (rows[l].to(torch.int64) + first).to(torch.uint32)
        assert int(far.cpu().numpy().max()) == 2 ** 32 - 1
        raw = fmmds.TreeC()
        C.memmove(C.byref(raw), C.byref(tree.raw), C.sizeof(raw))
        getattr(raw, lists + "_off")[l] = far.data_ptr()
        getattr(raw, lists + "_idx")[l] = entries_at_end.data_ptr()
        moved = fmmds.Tree(tree.L, 0, tree.src, tree.recv, tree.nnz_e2, tree.nnz_e4, {}, {}, {}, {})
        moved.raw = raw
        got = ctx.box_types(moved, lpar, owner, 1)
        torch.cuda.synchronize()
        kept.append(far)
        for k in want:
            assert torch.equal(got[k], want[k]), (l, k)
    ctx.close()
    del entries_at_end, kept
    torch.cuda.empty_cache()
