"""Batched builds of fixed-depth sets next to cluster-size sets, where a fixed-depth
set has a sub-cell too full for one block: the call builds that set by the radix
passes and returns every tree, from device and from host memory, the first time and
again.  Bit for bit against the oracle."""
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


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("L", [0, 4, 9])
def test_full_fixed_depth_set_next_to_cluster_size_sets(ctx, orc, L, host):
    full = workloads.clumps(50000, 1, nclumps=1, sigma=0.005)
    u, c = workloads.uniform(20001, 2), workloads.clumps(30000, 3, nclumps=2, sigma=0.002)
    sets, levels = [(full, full), (u, u), (c, u)], [L, None, None]

    def tensor(a):
        t = torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32))
        return t if host else t.cuda()

    kept = {id(a): tensor(a) for a in (full, u, c)}
    pairs = [(kept[id(a)], kept[id(b)]) for a, b in sets]
    want = [orc.build_tree(a, b, L=v) if v is not None else orc.build_tree(a, b, s=64)
            for (a, b), v in zip(sets, levels)]
    for _ in range(2):
        trees = ctx.build_batched(pairs, s=64, levels=levels,
                                  flags=fmmds.FMM_FLAG_HOST_INPUT if host else 0)
        for t, w in zip(trees, want):
            assert t.L == w["L"]
            compare_full(t.numpy(), w, t.L)
