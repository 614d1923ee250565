"""Points outside the cube in a few of many bucket tiles, which other tiles of the
launch see while they start: the call returns the domain error, and the context
builds the repaired points right afterwards."""
import numpy as np
import pytest

from paper_1301_1704_gb300 import fmmds, workloads
from tests.test_gpu_parity import compare_full

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [70001, 3000000])
@pytest.mark.parametrize("bad", [float("nan"), -1e-7, 1.0000002, float("inf")])
def test_bad_points_in_some_tiles(orc, n, bad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1301_1704_gb300 import build
    build.build()
    ctx = fmmds.Context(0)
    pts = workloads.uniform(n, 41)
    good = torch.from_numpy(pts).cuda()
    broken = good.clone()
    broken[:: n // 9, 1] = bad
    want = orc.build_tree(pts, pts, L=4, parallel=True)
    for _ in range(2):
        with pytest.raises(fmmds.FmmError) as e:
            ctx.build(broken, broken, L=4)
        assert e.value.code == fmmds.FMM_ERR_DOMAIN
        compare_full(ctx.build(good, good, L=4).numpy(), want, 4)
    ctx.close()
