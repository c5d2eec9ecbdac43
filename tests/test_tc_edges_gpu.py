"""Tensor-core path at the edges of its tiles: columns outside the volume (its converters repeat the
first and last column by groups of four), one row and one plane, planes fewer than the converter
groups, several items per CTA and a batch in one launch, against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import run_gpu

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2203_10213_gb300 as vkt  # noqa: E402

# of sum|w| max|x|: two 11-bit halves of each factor and the product of the low halves left out
# (3 * 2^-22), at most 27 truncated sums a plane (2^-23 each) and k rounded ones over the planes
TOL = 2.0 ** -18


def check(got, src, w):
    ref = oracle.correlate(src, w.astype(np.float64))
    scale = np.abs(w).astype(np.float64).sum() * np.abs(src).max()
    assert np.abs(got.astype(np.float64) - ref).max() <= TOL * scale


@pytest.mark.parametrize("k", [5, 7, 9])
@pytest.mark.parametrize("shape", [(1, 1, 4), (2, 128, 16), (3, 129, 20), (1, 256, 12), (5, 127, 44), (4, 3, 32)])
def test_edges(k, shape):
    r = np.random.RandomState(k + shape[2])
    src = r.uniform(-1, 1, shape).astype(np.float32)
    w = r.standard_normal((k, k, k)).astype(np.float32)
    check(run_gpu(vkt, src, vkt.Filter.dense(w), torch.float32, path="tensor"), src, w)


def test_many_items_per_cta():
    # 13 x 1 tiles, more chunks than SMs in all
    r = np.random.RandomState(3)
    src = r.uniform(-1, 1, (150, 20, 200)).astype(np.float32)
    w = r.standard_normal((7, 7, 7)).astype(np.float32)
    check(run_gpu(vkt, src, vkt.Filter.dense(w), torch.float32, path="tensor"), src, w)


@pytest.mark.parametrize("k", [5, 7, 9])
def test_batch_in_one_launch(k, capfd):
    r = np.random.RandomState(k)
    src = r.uniform(-1, 1, (3, 11, 40, 36)).astype(np.float32)
    w = r.standard_normal((k, k, k)).astype(np.float32)
    with vkt.policy(debug=vkt.DEBUG_LOG):
        out = vkt.apply_filter_autograd(torch.from_numpy(src).cuda(), torch.from_numpy(w).cuda(), "tensor")
    torch.cuda.synchronize()
    vkt.synchronize()
    assert capfd.readouterr().err.count("[vkt] tensor") == 1
    for i in range(3):
        check(out[i].cpu().numpy(), src[i], w)
