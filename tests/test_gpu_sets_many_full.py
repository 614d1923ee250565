"""One call with more fixed-depth sets than blocks of the plan kernel are resident at
once, a third of them with a sub-cell too full for one block, among sets that fit and
empty ones: every set's tree, bit for bit against the oracle, the first time (the
build starts again with the full sets on the radix path) and again."""
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


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


@pytest.mark.parametrize("sets,L", [(600, 3), (310, 6)])
def test_many_full_sets(ctx, orc, sets, L):
    rng = np.random.default_rng(sets)
    pts = []
    for i in range(sets):
        if i % 3 == 1:  # more points in one octant than a block sorts
            pts.append(workloads.clumps(int(rng.integers(6600, 9000)), i, nclumps=1, sigma=1e-4))
        else:
            pts.append(workloads.uniform(int(rng.integers(0, 900)), i))
    devs = [_dev(p) for p in pts]
    want = [orc.build_tree(p, p, L=L) for p in pts]
    for _ in range(2):
        for t, w in zip(ctx.build_batched([(d, d) for d in devs], L=L), want):
            compare_full(t.numpy(), w, L)
