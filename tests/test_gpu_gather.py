"""Alg. 2 over a level at the run lengths where the copy changes course: runs that
fill, straddle and leave over parts of the 32 floats a warp writes at a time,
receivers with few and no neighbours, and a run too long for 32-bit counts."""
import numpy as np
import pytest

from paper_1301_1704_gb300 import workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1301_1704_gb300 import build, fmmds
    build.build()
    c = fmmds.Context(0)
    yield c
    c.close()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


@pytest.mark.parametrize("per_box", [1, 2, 11, 32, 33])
@pytest.mark.parametrize("share", [0.1, 1.0])
def test_run_lengths(ctx, orc, per_box, share):
    from paper_1301_1704_gb300 import fmmds
    rng = np.random.default_rng(per_box)
    cells = workloads.lattice(3)
    cells = cells[rng.random(len(cells)) < share]
    src = np.repeat(cells, per_box, axis=0) + (rng.random((len(cells) * per_box, 3)) - 0.5) / 16
    src = np.ascontiguousarray(src, dtype=np.float32)
    recv = workloads.uniform(900, 5)
    tree = ctx.build(_dev(src), _dev(recv), L=3, flags=fmmds.FMM_FLAG_SORTED_XYZ)
    want = orc.build_tree(src, recv, L=3)
    off, pts = ctx.gather_e2(tree, 3)
    woff, wpts = orc.gather_e2(want, src, 3)
    assert np.array_equal(off.cpu().numpy().view(np.uint32).astype(np.uint64), woff)
    assert np.array_equal(pts.cpu().numpy(), wpts)


def test_one_long_run(ctx):
    from paper_1301_1704_gb300 import fmmds
    n = (1 << 24) + 5
    gen = torch.Generator(device="cuda").manual_seed(3)
    src = 0.3 + 0.1 * torch.rand((n, 3), generator=gen, device="cuda")
    recv = torch.tensor([[0.35, 0.35, 0.35], [0.9, 0.9, 0.9]], device="cuda")
    tree = ctx.build(src, recv, L=2, flags=fmmds.FMM_FLAG_SORTED_XYZ)
    off, pts = ctx.gather_e2(tree, 2)
    assert tree.src.nbox[2] == 1 and off.tolist() == [0, n, n]
    assert torch.equal(pts, tree.sorted_src)
