"""The renderer's pixel tiles and kept cells: views along every axis, each way up, and oblique ones,
against the oracle (the tile and the kept cell depend on the view)."""
import os
import sys

import numpy as np
import pytest
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import oracle  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    import paper_2203_10213_gb300 as vkt

LUT = np.array([[0, 0, 0.2, 0.0], [0.2, 0.5, 0.8, 0.02], [1, 0.8, 0.4, 0.15]], np.float32)
# eye relative to the volume's size, up
VIEWS = [((0.5, 0.6, -1.2), (0, 1, 0)), ((0.5, 0.6, -1.2), (1, 0, 0)), ((-1.2, 0.6, 0.5), (0, 1, 0)),
         ((-1.2, 0.6, 0.5), (0, 0, 1)), ((0.5, -1.2, 0.6), (0, 0, 1)), ((0.5, -1.2, 0.6), (1, 0, 0)),
         ((-0.6, -0.5, -0.55), (0, 1, 0)), ((0.4, 0.45, 0.5), (0.3, 1, 0))]


@pytest.mark.parametrize("view", range(len(VIEWS)))
@pytest.mark.parametrize("fmt", [synth.U8, synth.U16, synth.F32])
def test_views_match_oracle(view, fmt):
    shape = (36, 28, 44)
    v = synth.volume("blobs", fmt, tuple(reversed(shape)), 77)
    n = np.array([shape[2], shape[1], shape[0]], np.float64)
    (eye, up), center = VIEWS[view], 0.5 * n + np.array([0.3, -0.2, 0.1])
    eye = np.array(eye) * n
    args = [tuple(float(np.float32(x)) for x in a) for a in (eye, center, up)]
    for step in (0.5, 1.25):
        got = vkt.render(torch.from_numpy(v).cuda(), 61, 45, *args, 0.9, step, LUT).cpu().numpy()
        vkt.synchronize()
        ref = oracle.render(v, 0.0, 1.0, 61, 45, *args, float(np.float32(0.9)), step, 2.0, (0, 0, 0, 0), LUT)
        # float32 positions may put a ray's last sample on the other side of the box's face: one
        # sample's opacity, 1 - 0.85^1.25, in the few rays whose length is that near to whole steps
        err = np.abs(got - ref).max(axis=-1)
        assert np.mean(err > 2e-4) < 0.01, float(np.mean(err > 2e-4))
        assert err.max() < 0.19, float(err.max())
