"""Which path a dense k = 5 filter of float32 volumes takes by rule, alone and in a batch: sizes on
either side of the line, one volume the same way through both entry points, and batches whose spacing no
tensor map describes."""
import ctypes

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

import paper_2203_10213_gb300 as vkt  # noqa: E402
from gpu_util import compare  # noqa: E402

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

W = np.random.RandomState(2).standard_normal((5, 5, 5)).astype(np.float32)


@pytest.fixture(autouse=True)
def by_rule():
    """The rule alone: no measured choices."""
    was = ctypes.c_int32()
    vkt.check(vkt._lib.vktAutotuneGetEnabled(ctypes.byref(was)))
    vkt.check(vkt._lib.vktAutotuneSetEnabled(0))
    yield
    vkt.check(vkt._lib.vktAutotuneSetEnabled(was.value))


def volumes(n, shape, gap=0):
    """n volumes of one buffer, `gap` voxels between them, and as many destinations."""
    size = int(np.prod(shape))
    r = np.random.RandomState(size % 1000 + n)
    x = torch.from_numpy(r.random_sample((n, size + gap)).astype(np.float32)).cuda()
    return [t[:, :size].unflatten(1, shape) for t in (x, torch.zeros_like(x))]


def paths(capfd, call):
    capfd.readouterr()
    with vkt.policy(debug=True):
        call()
    vkt.synchronize()
    log = capfd.readouterr().err
    return log.count("[vkt] tensor k=5"), log.count("[vkt] direct k=5")


# n, (nz, ny, nx), launches on the tensor and on the direct path
@pytest.mark.parametrize("n,shape,want", [(1, (64, 64, 64), (0, 1)), (2, (32, 32, 32), (0, 1)),
                                          (4, (64, 64, 64), (0, 1)), (1, (128, 128, 128), (1, 0)),
                                          (8, (128, 128, 128), (1, 0)), (4, (96, 100, 132), (1, 0)),
                                          (8, (128, 32, 160), (0, 1)), (1, (96, 100, 132), (1, 0))])
def test_path_by_rule(n, shape, want, capfd):
    x, y = volumes(n, shape)
    filt = vkt.Filter.dense(W)
    vx, vy = ([vkt.StructuredVolume.from_tensor(t[i]) for i in range(n)] for t in (x, y))
    assert paths(capfd, lambda: vkt.apply_filter_batch(vy, vx, [filt] * n)) == want
    batch = y.clone()
    if n == 1:
        assert paths(capfd, lambda: vkt.apply_filter(vy[0], vx[0], filt)) == want
        assert torch.equal(y, batch)
    for i in (0, n - 1):
        src = x[i].cpu().numpy()
        compare(batch[i].cpu().numpy(), oracle.correlate(src, W, 0.0, 1.0), W, src, (0, 1), (0, 1), f"{n} {shape} {i}")


def test_spacing_without_a_tensor_map(capfd):
    x, y = volumes(3, (96, 100, 132), gap=2)
    filt = vkt.Filter.dense(W)
    vx, vy = ([vkt.StructuredVolume.from_tensor(t[i]) for i in range(3)] for t in (x, y))
    assert paths(capfd, lambda: vkt.apply_filter_batch(vy, vx, [filt] * 3)) == (0, 1)
    src = x[2].cpu().numpy()
    compare(y[2].cpu().numpy(), oracle.correlate(src, W, 0.0, 1.0), W, src, (0, 1), (0, 1), "spacing")
