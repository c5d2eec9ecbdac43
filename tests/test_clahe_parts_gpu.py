"""CLAHE with 1, 2, 4 and 8 CTAs to a brick, as the log says, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2203_10213_gb300 as vkt  # noqa: E402


# brick (x, y, z), bricks per axis, CTAs to a brick: one more doubling from 8192 voxels on, while the
# grid is resident; loads of 16, 4 and 1 bytes
@pytest.mark.parametrize("brick,bricks,parts", [((32, 32, 7), (2, 2, 2), 1), ((32, 32, 8), (2, 2, 2), 2),
                                                ((36, 30, 9), (2, 1, 2), 2), ((33, 31, 15), (1, 2, 2), 2),
                                                ((32, 32, 16), (2, 2, 2), 4), ((31, 35, 17), (2, 1, 1), 4),
                                                ((32, 32, 32), (2, 1, 2), 8), ((16, 16, 32), (8, 8, 10), 1)])
def test_ctas_per_brick(brick, bricks, parts, capfd):
    shape = tuple(reversed([s * n for s, n in zip(brick, bricks)]))
    v = (np.random.RandomState(sum(shape)).beta(2, 5, shape) * 255).astype(np.uint8)
    src = torch.from_numpy(v).cuda()
    capfd.readouterr()
    with vkt.policy(debug=True):
        got = vkt.clahe3d(src, bricks, 2.0)
    vkt.synchronize()
    assert f", {parts} CTAs per brick" in capfd.readouterr().err
    ref, t, _ = oracle.clahe3d(v, bricks, 2.0)
    # within 1e-3 of a tie either neighbour is right
    clear = np.abs(t - np.floor(t) - 0.5) > 1e-3
    np.testing.assert_array_equal(got.cpu().numpy()[clear], ref[clear])
