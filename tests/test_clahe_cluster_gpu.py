"""CLAHE where several CTAs of a cluster share a brick's histogram (few large bricks): against the
oracle, with rows read as vectors and voxel by voxel, and a flat volume, whose counts all meet in
one bin."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2203_10213_gb300 as vkt  # noqa: E402


# (nz, ny, nx), bricks (x, y, z): 2, 4 and 8 CTAs to a brick
@pytest.mark.parametrize("shape,bricks", [((32, 32, 64), (2, 1, 2)), ((64, 64, 64), (2, 2, 2)),
                                          ((65, 50, 70), (1, 1, 1)), ((48, 40, 66), (1, 2, 1))])
@pytest.mark.parametrize("flat", [False, True])
def test_shared_bricks(shape, bricks, flat):
    r = np.random.RandomState(sum(shape))
    v = np.full(shape, 37, np.uint8) if flat else (r.beta(2, 5, shape) * 255).astype(np.uint8)
    got = vkt.clahe3d(torch.from_numpy(v).cuda(), bricks, 2.0)
    torch.cuda.synchronize()
    vkt.synchronize()
    ref, t, _ = oracle.clahe3d(v, bricks, 2.0)
    # within 1e-3 of a tie either neighbour is right
    clear = np.abs(t - np.floor(t) - 0.5) > 1e-3
    np.testing.assert_array_equal(got.cpu().numpy()[clear], ref[clear])
