"""The list kernels at the sizes where they change course: chunks of four parents
with a ragged end, levels spread one parent a warp, parents with few and with
eight receiver children, with short and with long candidate lists, and jobs of
a batch without receivers or sources.  Bit for bit against the oracle."""
import numpy as np
import pytest

from paper_1301_1704_gb300 import workloads
from tests.test_gpu_parity import compare_full

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


def _subset(level, share, seed):
    """Centres of a random share of a level's boxes."""
    p = workloads.lattice(level)
    keep = np.random.default_rng(seed).random(len(p)) < share
    keep[0] = True
    return np.ascontiguousarray(p[keep])


@pytest.mark.parametrize("share", [0.002, 0.05, 0.3, 0.7, 1.0])
@pytest.mark.parametrize("L", [2, 3, 5, 6])
def test_box_occupancies(ctx, orc, L, share):
    src, recv = _subset(L, share, 10 * L), _subset(L, 1.0 - 0.5 * share, 10 * L + 1)
    for a, b in ((src, recv), (recv, src)):
        compare_full(ctx.build(_dev(a), _dev(b), L=L).numpy(), orc.build_tree(a, b, L=L), L)


@pytest.mark.parametrize("m", [1, 4863, 4864, 4865, 4872])
def test_one_launch_or_two(ctx, orc, m):
    """Around the parents that one launch a level takes (608 blocks of eight)."""
    src, recv = workloads.uniform(6000, 3), workloads.uniform(m, m)
    compare_full(ctx.build(_dev(src), _dev(recv), L=7).numpy(), orc.build_tree(src, recv, L=7), 7)


def test_jobs_without_points(ctx, orc):
    none = np.zeros((0, 3), np.float32)
    pairs = [(_subset(4, 0.4, k), _subset(4, 0.6, 50 + k)) for k in range(7)]
    pairs[0] = (none, pairs[0][1])
    pairs[3] = (pairs[3][0], none)
    pairs[6] = (none, none)
    levels = [4, 2, 5, 4, 1, 3, 4]
    trees = ctx.build_batched([(_dev(a), _dev(b)) for a, b in pairs], levels=levels)
    for (a, b), L, t in zip(pairs, levels, trees):
        compare_full(t.numpy(), orc.build_tree(a, b, L=L), L)
