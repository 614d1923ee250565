"""Cluster-size pairs whose sets are too full at their first sort depth: a little, by
eight and by more, with repeated points (no depth is enough), next to a set that
is not, shared between pairs, and in the box-key order.  Bit for bit against the
oracle."""
import numpy as np
import pytest

from paper_1301_1704_gb300 import fmmds, workloads
from tests.test_gpu_parity import compare_full

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CLUMPS = [(3000, 0.02), (40000, 0.01), (40000, 0.0005), (300000, 0.01), (300000, 0.001)]


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


@pytest.mark.parametrize("s", [3, 64, 700])
@pytest.mark.parametrize("n,sigma", CLUMPS)
def test_clumps_with_a_uniform_partner(ctx, orc, n, sigma, s):
    a, b = workloads.clumps(n, n, nclumps=3, sigma=sigma), workloads.uniform(n // 3 + 1, n + 1)
    for src, recv in ((a, b), (b, a)):
        want = orc.build_tree(src, recv, s=s)
        got = ctx.build(_dev(src), _dev(recv), s=s)
        assert got.L == want["L"]
        compare_full(got.numpy(), want, got.L)


def test_shared_partner_and_repeated_points(ctx, orc):
    u, c1 = workloads.uniform(5000, 1), workloads.clumps(30000, 2, nclumps=2, sigma=0.002)
    rep = np.repeat(workloads.uniform(40, 3), 50, axis=0)
    du, d1, dr = _dev(u), _dev(c1), _dev(rep)
    pairs = [(u, c1), (c1, u), (u, u), (rep, u)]
    trees = ctx.build_batched([(du, d1), (d1, du), (du, du), (dr, du)], s=20)
    for (src, recv), t in zip(pairs, trees):
        want = orc.build_tree(src, recv, s=20)
        assert t.L == want["L"]
        compare_full(t.numpy(), want, t.L)


def test_box_key_order(ctx, orc):
    a, b = workloads.clumps(40000, 9, nclumps=2, sigma=0.003), workloads.uniform(9000, 10)
    want = orc.build_tree(a, b, s=16, order=orc.ORDER_BOX)
    got = ctx.build(_dev(a), _dev(b), s=16, flags=fmmds.FMM_FLAG_BOX_ORDER)
    assert got.L == want["L"]
    compare_full(got.numpy(), want, got.L)
