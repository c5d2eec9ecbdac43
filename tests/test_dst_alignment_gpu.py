"""Destinations that start on a voxel boundary but not on 16 bytes: the stores are as wide as the
address allows, and nothing outside the volume is written."""
import os
import sys

import numpy as np
import pytest
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    import paper_2203_10213_gb300 as vkt


@pytest.mark.parametrize("offset", [1, 2, 3])
@pytest.mark.parametrize("src", [torch.uint8, torch.uint16, torch.float32])
@pytest.mark.parametrize("dst", [torch.uint8, torch.uint16, torch.float32])
def test_unaligned_destination(offset, src, dst):
    shape = (6, 21, 136)
    n = int(np.prod(shape))
    g = torch.Generator().manual_seed(3)
    if src == torch.float32:
        s = torch.rand(shape, generator=g).cuda()
    else:
        s = torch.randint(0, 256, shape, generator=g).to(torch.int32).to(src).cuda()
    laplace = np.zeros((3, 3, 3), np.float32)
    laplace[1, 1, 1] = -6
    laplace[0, 1, 1] = laplace[2, 1, 1] = laplace[1, 0, 1] = laplace[1, 2, 1] = laplace[1, 1, 0] = laplace[1, 1, 2] = 1
    box = np.full((3, 3, 3), 1 / 27, np.float32)
    for filt in (vkt.Filter.gaussian(3, 1.0), vkt.Filter.gaussian(5, 1.5), vkt.Filter.gaussian(7, 2.0),
                 vkt.Filter.dense(laplace), vkt.Filter.dense(box)):
        want = torch.zeros(shape, dtype=dst, device="cuda")
        vkt.filter_tensor(s, filt, out=want, dst_range=(-1.0, 1.0))
        raw = torch.full((n + 16,), 7, dtype=torch.int32).to(dst).cuda()
        vkt.filter_tensor(s, filt, out=raw[offset:offset + n].view(shape), dst_range=(-1.0, 1.0))
        torch.cuda.synchronize()
        vkt.synchronize()
        got, ref = raw.cpu().numpy(), want.cpu().numpy().reshape(-1)
        np.testing.assert_array_equal(got[offset:offset + n], ref)
        assert (got[:offset] == 7).all() and (got[offset + n:] == 7).all()
