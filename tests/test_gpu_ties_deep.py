"""Repeated points where the radix passes sort every key bit: trees of 19 to 21
levels, and the partner of a set whose cluster size no level meets.  Points with
equal keys stay in the order of their indices.  Bit for bit against the oracle."""
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


def _repeated(distinct, copies, seed):
    pts = np.repeat(workloads.uniform(distinct, seed), copies, axis=0)
    return pts[np.random.default_rng(seed).permutation(len(pts))]


@pytest.mark.parametrize("kind", [fmmds.FMM_SORT_RTS, fmmds.FMM_SORT_ONESWEEP, fmmds.FMM_SORT_BUCKET])
@pytest.mark.parametrize("L", [18, 19, 20, 21])
@pytest.mark.parametrize("distinct,copies", [(40, 100), (2000, 5)])
def test_deep_trees(ctx, orc, kind, L, distinct, copies):
    a, b = _repeated(distinct, copies, 31), _repeated(copies, distinct, 32)
    ctx.set_tuning(kind)
    compare_full(ctx.build(_dev(a), _dev(b), L=L).numpy(), orc.build_tree(a, b, L=L), L)


def test_partner_of_an_unmet_cluster_size(ctx, orc):
    a, b = _repeated(1, 100, 33), _repeated(2000, 5, 34)
    for src, recv in ((a, b), (b, a)):
        want = orc.build_tree(src, recv, s=8)
        got = ctx.build(_dev(src), _dev(recv), s=8).numpy()
        assert (got["L"], got["s_unmet"]) == (want["L"], want["s_unmet"]) == (21, 1)
        compare_full(got, want, 21)
