"""Coarser boxes of radix-path sets, eight boxes a thread and two: every bound on the
depth the kernel is compiled for, tiles with remainders and whole ones, next to a
set whose capacity decides how many boxes a thread takes.  Bit for bit against the
oracle."""
import numpy as np
import pytest

from paper_1301_1704_gb300 import workloads
from tests.test_gpu_parity import compare_full

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SORT_RTS = 0
SIZES = (1, 7, 9, 1023, 1025, 4096, 4097, 20003)


@pytest.mark.parametrize("big", [0, 4_300_000])
@pytest.mark.parametrize("depth", [1, 8, 9, 12, 13, 16, 17, 21])
def test_tiles_and_depths(orc, big, depth):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1301_1704_gb300 import build, fmmds
    build.build()
    ctx = fmmds.Context(0)
    ctx.set_tuning(SORT_RTS)
    pts = [workloads.uniform(n, 100 + n) if n % 2 else workloads.clumps(n, n, nclumps=3, sigma=0.02)
           for n in SIZES]
    levels = [max(depth - (i % 3), 1) for i in range(len(pts))]
    levels[-2] = levels[-1] = depth
    if big:  # 4.3e6 level-8 boxes at most: eight boxes a thread for every set
        pts.append(workloads.sphere(big, 5, radius=0.05))
        levels.append(8)
    devs = [torch.from_numpy(np.ascontiguousarray(p, dtype=np.float32)).cuda() for p in pts]
    trees = ctx.build_batched([(d, d) for d in devs], levels=levels)
    for p, L, t in list(zip(pts, levels, trees))[:len(SIZES)]:
        compare_full(t.numpy(), orc.build_tree(p, p, L=L), L)
    ctx.close()
