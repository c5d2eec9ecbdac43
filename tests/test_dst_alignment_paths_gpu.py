"""Float32 destinations off 16 bytes on the paths that test_dst_alignment_gpu.py does not take: other
filter sizes, regions, batches (each volume's own start, and a spacing off 16 bytes) and gradients.  The
values are those of an aligned destination, and nothing outside the volume is written."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2203_10213_gb300 as vkt  # noqa: E402

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def dense(k):
    return vkt.Filter.dense(np.random.RandomState(k).standard_normal((k, k, k)).astype(np.float32))


def source(shape, dtype, seed=3):
    g = torch.Generator().manual_seed(seed)
    return (torch.rand(shape, generator=g) if dtype == torch.float32 else
            torch.randint(0, 256, shape, generator=g).to(torch.int32).to(dtype)).cuda()


def off(n, offset, fill=7.0):
    """A buffer, and the n floats that start `offset` floats after a 16-byte boundary."""
    raw = torch.full((n + 16,), fill, device="cuda")
    return raw, raw[offset:offset + n]


def same(raw, offset, want):
    got, n = raw.cpu().numpy(), want.numel()
    np.testing.assert_array_equal(got[offset:offset + n], want.cpu().numpy().reshape(-1))
    assert (got[:offset] == 7).all() and (got[offset + n:] == 7).all()


@pytest.mark.parametrize("offset", [1, 2, 3])
@pytest.mark.parametrize("dtype", [torch.uint8, torch.uint16, torch.float32])
@pytest.mark.parametrize("nx", [136, 139])
@pytest.mark.parametrize("region", [False, True])
def test_filters(offset, dtype, nx, region):
    shape = (11, 21, nx)
    src = source(shape, dtype)
    roi = ((4, 3, 2), (nx - 5, 18, 9)) if region else None
    for filt in (vkt.Filter.gaussian(1, 1.0), vkt.Filter.gaussian(3, 1.0), vkt.Filter.gaussian(5, 1.5),
                 vkt.Filter.gaussian(9, 2.0), dense(1), dense(3), dense(5), dense(7)):
        want = torch.full(shape, 7.0, device="cuda")
        vkt.filter_tensor(src, filt, out=want, roi=roi)
        raw, out = off(want.numel(), offset)
        vkt.filter_tensor(src, filt, out=out.view(shape), roi=roi)
        vkt.synchronize()
        same(raw, offset, want)


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_separable_batch(offset):
    shapes = [(9, 20, 40), (6, 33, 72), (17, 5, 30), (8, 40, 64)]
    dtypes = [torch.uint8, torch.float32, torch.uint16, torch.float32]
    for k in (1, 3, 5, 7):
        srcs = [source(s, d, i) for i, (s, d) in enumerate(zip(shapes, dtypes))]
        filt = vkt.Filter.gaussian(k, 1.0)
        want = [torch.zeros(s, device="cuda") for s in shapes]
        bufs = [off(w.numel(), offset) for w in want]
        vs = [vkt.StructuredVolume.from_tensor(s) for s in srcs]
        for dsts in (want, [b[1].view(s) for b, s in zip(bufs, shapes)]):
            vkt.apply_filter_batch([vkt.StructuredVolume.from_tensor(d) for d in dsts], vs, [filt] * len(vs))
        vkt.synchronize()
        for (raw, _), w in zip(bufs, want):
            same(raw, offset, w)


# (the volumes of a batch stand `gap` floats apart, the first one on 16 bytes)
@pytest.mark.parametrize("gap", [1, 2, 3])
@pytest.mark.parametrize("shape", [(10, 17, 40), (64, 512, 128)])
def test_spaced_batch_and_gradients(gap, shape):
    n, size = 3, int(np.prod(shape))
    filt = dense(3)
    x, gy = source((n,) + shape, torch.float32), source((n,) + shape, torch.float32, 5)
    vx, vgy = ([vkt.StructuredVolume.from_tensor(t[i]) for i in range(n)] for t in (x, gy))
    want = [torch.zeros(shape, device="cuda") for _ in range(n)]
    for i in range(n):
        vkt.apply_filter(vkt.StructuredVolume.from_tensor(want[i]), vx[i], filt, path="direct")
    wide, spaced = torch.zeros((n,) + shape, device="cuda"), torch.zeros(n, size + gap, device="cuda")
    outs = [spaced[i, :size].view(shape) for i in range(n)]
    with vkt.policy(path="direct"):
        vkt.apply_filter_batch([vkt.StructuredVolume.from_tensor(o) for o in outs], vx, [filt] * n)
    vkt.synchronize()
    for i in range(n):
        np.testing.assert_array_equal(outs[i].cpu().numpy(), want[i].cpu().numpy())
    vkt.apply_filter_backward_batch([vkt.StructuredVolume.from_tensor(wide[i]) for i in range(n)], None, vgy, vx, filt)
    spaced.zero_()
    vkt.apply_filter_backward_batch([vkt.StructuredVolume.from_tensor(o) for o in outs], None, vgy, vx, filt)
    vkt.synchronize()
    assert not spaced[:, size:].cpu().numpy().any()
    for i in range(n):
        # (the shell's shares are added to the face voxels atomically, in any order)
        np.testing.assert_allclose(outs[i].cpu().numpy(), wide[i].cpu().numpy(), rtol=0, atol=1e-4)
