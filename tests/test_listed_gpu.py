"""Dense filters over integer sources into integer codes by the listed modes of the direct kernel:
one float32 weight per tap (uint8 codes) and high and low weights (uint16 codes)."""
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

DT = {synth.U8: torch.uint8, synth.U16: torch.uint16}
QMAX = {synth.U8: 255.0, synth.U16: 65535.0}
# (nz, ny, nx): tensor map, row copies, tile edges, thinner than the filter
SHAPES = [(9, 17, 64), (21, 66, 136), (13, 16, 65), (3, 2, 8), (1, 1, 1), (40, 18, 24)]


def codes(seed, shape, sfmt):
    r = np.random.RandomState(seed)
    return r.randint(0, int(QMAX[sfmt]) + 1, shape).astype(np.uint8 if sfmt == synth.U8 else np.uint16)


def run(src, filt, dfmt, drange=(0.0, 1.0), roi=None, offset=0):
    flat = torch.empty(src.size + offset, dtype=torch.uint8 if src.dtype == np.uint8 else torch.uint16)
    flat[offset:] = torch.from_numpy(src.reshape(-1))
    t = flat.cuda()[offset:].view(src.shape)
    out = torch.zeros(src.shape, dtype=DT[dfmt], device="cuda")
    vkt.filter_tensor(t, filt, out=out, dst_range=drange, path="direct", roi=roi)
    torch.cuda.synchronize()
    vkt.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("sfmt", [synth.U8, synth.U16])
@pytest.mark.parametrize("k", [3, 5, 7, 9])
@pytest.mark.parametrize("offset", [0, 1])
def test_ties_round_to_even(sfmt, k, offset):
    """Weights that are multiples of 1/64 (sums exact in 64 bits): many results are exact ties.
    offset 1: the source is not 16-byte aligned (plain loads)."""
    r = np.random.RandomState(k)
    w = (r.randint(-3, 5, (k, k, k)) / 64.0).astype(np.float32)
    w[k // 2, k // 2, k // 2] += np.float32(1.0) - w.sum()
    for shape in SHAPES:
        src = codes(7 * k + sum(shape), shape, sfmt)
        got = run(src, vkt.Filter.dense(w), sfmt, offset=offset)
        v = oracle.correlate(src, w.astype(np.float64), 0.0, QMAX[sfmt])
        np.testing.assert_array_equal(got.astype(np.float64), np.clip(np.rint(v), 0, QMAX[sfmt]))


@pytest.mark.parametrize("sfmt,dfmt", [(synth.U8, synth.U8), (synth.U16, synth.U16), (synth.U8, synth.U16),
                                       (synth.U16, synth.U8)])
@pytest.mark.parametrize("k", [3, 5, 7, 9])
def test_random_weights_match_oracle(sfmt, dfmt, k):
    """Codes equal the 64-bit evaluation's wherever that is not within 1e-3 of a tie."""
    w = (np.random.RandomState(40 + k).standard_normal((k, k, k)) + 0.5)
    w = (w / w.sum()).astype(np.float32)
    drange = (-0.25, 1.5)
    for shape in SHAPES:
        src = codes(11 * k + sum(shape), shape, sfmt)
        got = run(src, vkt.Filter.dense(w), dfmt, drange)
        v = (oracle.correlate(src, w.astype(np.float64), 0.0, 1.0) - drange[0]) / (drange[1] - drange[0]) * QMAX[dfmt]
        clear = np.abs(v - np.floor(v) - 0.5) > 1e-3
        np.testing.assert_array_equal(got[clear], np.clip(np.rint(v), 0, QMAX[dfmt])[clear])


@pytest.mark.parametrize("sfmt", [synth.U8, synth.U16])
@pytest.mark.parametrize("drange", [(-1.0, 1.0), (-6.0, 6.0), (-1.0, 2.0)])
def test_laplacian_into_symmetric_range(sfmt, drange):
    """A signed destination range puts flat regions and every even sum on a tie; the codes are the
    compensated evaluation's, whose ties go to the even code."""
    w = synth.laplacian_3()
    for shape in SHAPES:
        src = codes(sum(shape), shape, sfmt)
        src[: shape[0] // 2] = 0
        got = run(src, vkt.Filter.dense(w), sfmt, drange)
        n = oracle.correlate(src, w.astype(np.float64), 0.0, QMAX[sfmt])      # whole numbers
        v = (n - drange[0] * QMAX[sfmt]) / (drange[1] - drange[0])
        want = np.clip(np.rint(v), 0, QMAX[sfmt])
        if drange[1] - drange[0] == 2.0:        # v is exact: ties are ties
            np.testing.assert_array_equal(got.astype(np.float64), want)
        else:
            clear = np.abs(v - np.floor(v) - 0.5) > 1e-3
            np.testing.assert_array_equal(got[clear], want[clear])


@pytest.mark.parametrize("sfmt", [synth.U8, synth.U16])
def test_region_equals_whole_volume(sfmt):
    shape, f = (21, 66, 136), vkt.Filter.dense(np.full((5, 5, 5), 0.008, np.float32))
    src = codes(5, shape, sfmt)
    whole, part = run(src, f, sfmt), run(src, f, sfmt, roi=((3, 2, 1), (70, 65, 17)))
    want = np.zeros_like(whole)
    want[1:17, 2:65, 3:70] = whole[1:17, 2:65, 3:70]
    np.testing.assert_array_equal(part, want)
