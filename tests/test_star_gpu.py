"""3^3 filters with taps on the axes only (vkt_star.cu) against the oracle: tile edges, every pair of
an integer source and a destination, one-sided taps, and the forms that stay with the general kernel."""
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

DT = {synth.U8: torch.uint8, synth.U16: torch.uint16, synth.F32: torch.float32}
QMAX = {synth.U8: 255.0, synth.U16: 65535.0}
# (nz, ny, nx): one lane, one tile, tile edges in x and y, several stages' worth of planes, thin
SHAPES = [(1, 1, 16), (3, 33, 128), (30, 31, 144), (9, 70, 272), (2, 2, 32)]


def star(taps):
    w = np.zeros((3, 3, 3), np.float32)
    w[0, 1, 1], w[1, 0, 1], w[1, 1, 0], w[1, 1, 1], w[1, 1, 2], w[1, 2, 1], w[2, 1, 1] = taps
    return w


FILTERS = {"laplacian": star((1, 1, 1, -6, 1, 1, 1)), "uneven": star((0.3, -0.7, 0.11, 0.9, 0.23, 0.05, -0.4)),
           "gradient": star((0, 0, -0.5, 0, 0.5, 0, 0)), "sharpen": star((-0.25, -0.25, -0.25, 2.5, -0.25, -0.25, -0.25))}


def run(src, w, dfmt, drange=(0.0, 1.0), roi=None, debug=False):
    t = torch.from_numpy(src).cuda()
    out = torch.zeros(src.shape, dtype=DT[dfmt], device="cuda")
    with vkt.policy(debug=vkt.DEBUG_LOG if debug else 0):
        vkt.filter_tensor(t, vkt.Filter.dense(w), out=out, dst_range=drange, path="direct", roi=roi)
    torch.cuda.synchronize()
    vkt.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("name", sorted(FILTERS))
@pytest.mark.parametrize("sfmt", [synth.U8, synth.U16])
@pytest.mark.parametrize("dfmt", [synth.U8, synth.U16, synth.F32])
def test_matches_oracle(name, sfmt, dfmt):
    w = FILTERS[name]
    for shape in SHAPES:
        r = np.random.RandomState(sum(shape))
        src = r.randint(0, int(QMAX[sfmt]) + 1, shape).astype(np.uint8 if sfmt == synth.U8 else np.uint16)
        ref = oracle.correlate(src, w.astype(np.float64), 0.0, 1.0)
        if dfmt == synth.F32:
            got = run(src, w, dfmt)
            # 7 products and sums of values up to 1, and the mapping
            assert np.abs(got - ref).max() <= 10 * 2.0 ** -24 * np.abs(w).sum()
        else:
            got = run(src, w, dfmt, (-1.0, 1.0))
            v = (ref + 1.0) / 2.0 * QMAX[dfmt]
            clear = np.abs(v - np.floor(v) - 0.5) > 1e-3
            np.testing.assert_array_equal(got[clear], np.clip(np.rint(v), 0, QMAX[dfmt])[clear])


def test_which_calls_take_it(capfd):
    w, r = FILTERS["laplacian"], np.random.RandomState(1)
    u8 = r.randint(0, 256, (8, 9, 32)).astype(np.uint8)
    diagonal = w.copy()
    diagonal[0, 0, 1] = 0.1
    infinite = w.copy()
    infinite[1, 1, 1] = np.inf
    for src, filt, roi, want in ((u8, w, None, True), (u8, diagonal, None, False), (u8, infinite, None, False),
                                 (u8, w, ((0, 0, 0), (32, 9, 7)), False), (u8[:, :, :30].copy(), w, None, False),
                                 (u8.astype(np.float32), w, None, False)):
        capfd.readouterr()
        run(src, filt, synth.F32, roi=roi, debug=True)
        assert ("direct-star" in capfd.readouterr().err) == want
