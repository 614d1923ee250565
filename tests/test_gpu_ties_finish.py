"""Points of one box whose low key bits agree in their top 32, and differ below, or not
at all: the finishing sort of the radix path orders them by the rest of the key, then
by index, at every sort depth.  Bit for bit against the oracle."""
import numpy as np
import pytest

from paper_1301_1704_gb300 import fmmds, workloads
from tests.test_gpu_parity import compare_full

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture()
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1301_1704_gb300 import build
    build.build()
    c = fmmds.Context(0)
    yield c
    c.close()


def _points(spots, copies, cells, seed):
    """`copies` points around each spot, `cells` cells of level 21 wide on every axis."""
    rng = np.random.default_rng(seed)
    at = np.floor(rng.random((spots, 1, 3)) * 2 ** 20)
    p = (at + rng.integers(0, cells, size=(spots, copies, 3))).reshape(-1, 3) / 2.0 ** 21
    return np.ascontiguousarray(p[rng.permutation(len(p))], dtype=np.float32)


@pytest.mark.parametrize("cells", [1, 2, 40, 5000])
@pytest.mark.parametrize("spots,copies", [(1, 2), (3, 33), (40, 250), (2500, 7)])
def test_close_points(ctx, orc, spots, copies, cells):
    a, b = _points(spots, copies, cells, spots + cells), workloads.uniform(100, 61)
    da, db = (torch.from_numpy(x).cuda() for x in (a, b))
    ctx.set_tuning(fmmds.FMM_SORT_RTS)
    for L in (0, 2, 5, 8, 10, 11, 14):
        compare_full(ctx.build(da, db, L=L).numpy(), orc.build_tree(a, b, L=L), L)
    want = orc.build_tree(a, b, s=copies)
    got = ctx.build(da, db, s=copies)
    assert got.L == want["L"]
    compare_full(got.numpy(), want, got.L)
