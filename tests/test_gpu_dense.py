"""Fixed-depth sets with a sub-cell too full for one block: the bucket path stops,
the set is built by radix passes to a depth that follows from its fullest
sub-cell, and the context goes there directly the next time.  Shallow and deep
trees, clumps, surfaces and one point repeated, next to sets that fit.  Bit for
bit against the oracle."""
import numpy as np
import pytest

from paper_1301_1704_gb300 import workloads
from tests.test_gpu_parity import compare_full

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture()
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


@pytest.mark.parametrize("n", [6200, 60001, 400003])
@pytest.mark.parametrize("L", [0, 2, 4, 7, 9])
def test_clump_next_to_sphere(ctx, orc, n, L):
    src = workloads.clumps(n, n, nclumps=1, sigma=0.01)
    recv = workloads.sphere(n // 2 + 1, n + 1, radius=0.1)
    s, r = _dev(src), _dev(recv)
    want = orc.build_tree(src, recv, L=L)
    for _ in range(2):
        compare_full(ctx.build(s, r, L=L).numpy(), want, L)


def test_repeated_point_and_batch(ctx, orc):
    pts = [np.repeat(np.array([[0.3, 0.7, 0.1]], np.float32), 9000, axis=0),
           workloads.uniform(30000, 2), workloads.clumps(50000, 3, nclumps=2, sigma=0.005)]
    devs, levels = [_dev(p) for p in pts], [5, 4, 3]
    for _ in range(2):
        for p, L, t in zip(pts, levels, ctx.build_batched([(d, d) for d in devs], levels=levels)):
            compare_full(t.numpy(), orc.build_tree(p, p, L=L), L)
