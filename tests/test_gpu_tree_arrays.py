"""The arrays of a tree are tensors of their own: an in-place change to one does not
count as a change to another (a saved index stays usable in a backward pass), saving
one writes that array alone, and the sources' and receivers' tensors of a set built
once are different objects over the same memory."""
import io

import numpy as np
import pytest

from paper_1301_1704_gb300 import fmmds, workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(params=[True, False], ids=["torch-allocator", "library-memory"])
def ctx(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1301_1704_gb300 import build
    build.build()
    c = fmmds.Context(0, torch_allocator=request.param)
    yield c
    c.close()


def _arrays(t):
    out = [x for sd in (t.src, t.recv) for x in [sd.perm, *sd.key, *sd.off, *sd.parent, *sd.child]]
    for d in (t.e2_off, t.e2_idx, t.e4_off, t.e4_idx):
        out += d.values()
    return [x for x in out if x.numel()]


def _tree(ctx, aliased):
    a = torch.from_numpy(workloads.uniform(3000, 5).astype(np.float32)).cuda()
    b = a if aliased else torch.from_numpy(workloads.uniform(2000, 6).astype(np.float32)).cuda()
    return ctx.build(a, b, L=3)


@pytest.mark.parametrize("aliased", [True, False])
def test_own_object_and_version(ctx, aliased):
    arrays = _arrays(_tree(ctx, aliased))
    assert len({id(x) for x in arrays}) == len(arrays)
    before = [x._version for x in arrays]
    arrays[0].add_(0)
    assert [x._version for x in arrays[1:]] == before[1:] and arrays[0]._version > before[0]


def test_shapes_types_and_storage(ctx):
    t = _tree(ctx, False)
    for x in _arrays(t):
        assert x.device == torch.device("cuda", 0) and x.is_contiguous() and not x.requires_grad
        assert x.storage_offset() == 0 and x.untyped_storage().nbytes() == x.numel() * x.itemsize
    assert all(k.dtype == torch.int64 for sd in (t.src, t.recv) for k in sd.key)
    assert t.src.perm.dtype == t.e4_idx[3].dtype == torch.int32
    assert t.src.perm.shape == (3000,) and t.recv.off[3].shape == (t.recv.nbox[3] + 1,)


def test_saved_index_survives_a_change_to_another_array(ctx):
    t = _tree(ctx, False)
    w = torch.ones(t.src.nbox[3], device="cuda", requires_grad=True)
    loss = w[t.e2_idx[3]].sum()
    t.src.perm.add_(1)
    loss.backward()
    idx = t.e2_idx[3].cpu().numpy()
    assert np.array_equal(w.grad.cpu().numpy(), np.bincount(idx, minlength=t.src.nbox[3]))


def test_save_writes_one_array(ctx):
    t = _tree(ctx, True)
    f = io.BytesIO()
    torch.save(t.src.perm, f)
    assert f.tell() < 4 * t.src.n + 4096
    f.seek(0)
    assert torch.equal(torch.load(f), t.src.perm)


def test_two_threads_and_contexts():
    """Trees built at the same time in two threads hold their own arrays."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import threading
    failed = []

    def work(n):
        c = fmmds.Context(0)
        a = torch.from_numpy(workloads.uniform(n, n).astype(np.float32)).cuda()
        for _ in range(30):
            t = c.build(a, a, L=4)
            sizes = [x.numel() for x in t.src.key + t.src.off + t.src.parent[1:]]
            want = list(t.src.nbox[:5])
            if sizes != want + [k + 1 for k in want] + want[1:]:
                failed.append(sizes)
            if not torch.equal(torch.sort(t.src.perm).values,
                               torch.arange(n, dtype=torch.int32, device="cuda")):
                failed.append(n)
        c.close()

    threads = [threading.Thread(target=work, args=(n,)) for n in (3000, 5001)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
