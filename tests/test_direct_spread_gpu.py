"""Direct launches of less than a wave take shared memory so that an SM holds no more CTAs than an even
spread needs: the launches say so, and the results are the oracle's, one CTA more than a round number per
SM and one less."""
import re

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")

import paper_2203_10213_gb300 as vkt  # noqa: E402
from gpu_util import compare  # noqa: E402

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


# (nz, ny, nx), k, source, destination: 1 to 3 CTAs per SM, with and without a tensor map, codes, Dot2
@pytest.mark.parametrize("shape,k,src,dst", [((60, 60, 61), 5, torch.uint16, torch.float32),
                                             ((100, 100, 99), 5, torch.uint16, torch.float32),
                                             ((151, 458, 45), 5, torch.uint16, torch.float32),
                                             ((64, 400, 64), 5, torch.uint8, torch.float32),
                                             ((128, 120, 128), 1, torch.uint8, torch.uint8),
                                             ((90, 64, 100), 5, torch.float32, torch.uint8),
                                             ((40, 70, 132), 3, torch.float32, torch.float32),
                                             ((33, 35, 37), 3, torch.uint8, torch.float32)])
def test_spread(shape, k, src, dst, capfd):
    r = np.random.RandomState(k + shape[0])
    v = r.random_sample(shape).astype(np.float32)
    if src != torch.float32:
        v = (v * (255 if src == torch.uint8 else 65535)).astype(np.uint8 if src == torch.uint8 else np.uint16)
    w = r.random_sample((k, k, k)).astype(np.float32)
    w = (w / w.sum(dtype=np.float64)).astype(np.float32)
    capfd.readouterr()
    with vkt.policy(debug=True, path="direct"):
        out = vkt.filter_tensor(torch.from_numpy(v).cuda(), vkt.Filter.dense(w), dst_dtype=dst)
    vkt.synchronize()
    log = capfd.readouterr().err
    grid, per_sm = re.search(r"grid=\((\d+),(\d+),(\d+)\).* per_sm=(\d+)", log).groups()[:3], int(
        re.search(r"per_sm=(\d+)", log).group(1))
    ctas = int(np.prod([int(x) for x in grid]))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert per_sm <= -(-ctas // sms)
    compare(out.cpu().numpy(), oracle.correlate(v, w, 0.0, 1.0), w, v, (0, 1), (0, 1), f"{shape} {k}")
