"""The kernels that march through the raw stages (separable: vkt_walk.cuh, dense 3^3 of float32:
vkt_march3.cu): bit-identical to the general kernels, which a call with a region of interest takes,
at tile edges, and which calls they take."""
import os
import sys

import numpy as np
import pytest
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import oracle  # noqa: E402

pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    import paper_2203_10213_gb300 as vkt

QMAX = {torch.uint8: 255, torch.uint16: 65535}


def source(shape, dtype, seed):
    r = np.random.RandomState(seed)
    if dtype == torch.float32:
        return r.standard_normal(shape).astype(np.float32)
    return r.randint(0, QMAX[dtype] + 1, shape).astype(np.uint8 if dtype == torch.uint8 else np.uint16)


def run(src, filt, dtype, roi=None, path="auto"):
    out = torch.zeros(src.shape, dtype=dtype, device="cuda")
    with vkt.policy(debug=vkt.DEBUG_LOG):
        vkt.filter_tensor(torch.from_numpy(src).cuda(), filt, out=out, path=path, roi=roi,
                          dst_range=(-1.0, 1.0) if dtype in QMAX else (0.0, 1.0))
    torch.cuda.synchronize()
    vkt.synchronize()
    return out.cpu().numpy()


def compare(src, filt, dtype, path, mark, capfd, rel):
    nz, ny, nx = src.shape
    capfd.readouterr()
    got = run(src, filt, dtype, path=path)
    assert mark in capfd.readouterr().err
    whole = run(src, filt, dtype, roi=((0, 0, 0), (nx, ny, nz - 1)), path=path)
    assert mark not in capfd.readouterr().err
    n = nz - 1
    np.testing.assert_array_equal(got[:n], whole[:n])
    if dtype == torch.float32:
        dense = filt.weights().astype(np.float64)
        ref = oracle.correlate(src, dense, 0.0, 1.0)
        assert np.abs(got - ref).max() <= rel * 2.0 ** -24 * np.abs(dense).sum() * max(np.abs(src).max(), 1.0)


# (nz, ny, nx): rows of whole 16 bytes around one and two tiles, one row, ragged y
F32 = [(3, 17, 36), (2, 16, 128), (2, 1, 132), (19, 33, 260)]


@pytest.mark.parametrize("k", [3, 5])
@pytest.mark.parametrize("shape", F32)
def test_separable_float32(k, shape, capfd):
    # one rounding per product and sum of the 3 passes of k taps
    compare(source(shape, torch.float32, k), vkt.Filter.gaussian(k, 1.1), torch.float32, "separable",
            "separable-walk", capfd, 3 * 2 * k)


@pytest.mark.parametrize("src", [torch.uint8, torch.uint16])
def test_separable_codes(src, capfd):
    compare(source((131, 301, 256), src, 4), vkt.Filter.gaussian(3, 1.0), torch.float32, "separable",
            "separable-walk", capfd, 20)


@pytest.mark.parametrize("shape", [(133, 305, 256), (200, 385, 260 - 68), (200, 401, 132 + 224)])
def test_dense_float32(shape, capfd):
    r = np.random.RandomState(6)
    filt = vkt.Filter.dense(r.uniform(-1, 1, (3, 3, 3)).astype(np.float32))
    compare(source(shape, torch.float32, 5), filt, torch.float32, "direct", "direct-march", capfd, 2 * 27)


def test_dense_float32_batch(capfd):
    # volumes of one allocation are one launch; each has its own faces
    src = source((4, 72, 272, 128), torch.float32, 7)
    w = np.random.RandomState(8).uniform(-1, 1, (3, 3, 3)).astype(np.float32)
    capfd.readouterr()
    with vkt.policy(debug=vkt.DEBUG_LOG):
        out = vkt.apply_filter_autograd(torch.from_numpy(src).cuda(), torch.from_numpy(w).cuda(), "direct")
    torch.cuda.synchronize()
    vkt.synchronize()
    assert "direct-march" in capfd.readouterr().err
    for i in range(4):
        np.testing.assert_array_equal(out[i].cpu().numpy(),
                                      run(src[i], vkt.Filter.dense(w), torch.float32, path="direct"))


def test_which_calls_take_it(capfd):
    dense = vkt.Filter.dense(np.random.RandomState(9).uniform(-1, 1, (3, 3, 3)).astype(np.float32))
    gauss = vkt.Filter.gaussian(3, 1.0)
    for shape, src, filt, path in (((9, 20, 32), torch.float32, gauss, "separable"),
                                   ((9, 20, 38), torch.float32, gauss, "separable"),
                                   ((9, 20, 256), torch.uint8, gauss, "separable"),
                                   ((9, 20, 128), torch.float32, dense, "direct"),
                                   ((133, 305, 144), torch.float32, dense, "direct")):
        capfd.readouterr()
        run(source(shape, src, 1), filt, torch.float32, path=path)
        err = capfd.readouterr().err
        assert "separable-walk" not in err and "direct-march" not in err
