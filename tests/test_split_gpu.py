"""Integer sources into integer codes by the split evaluation (vkt_sep_split.cuh): every way of
loading, tile edges, regions, and filters whose results lie on rounding ties."""
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
# (nz, ny, nx): rows of 16 bytes (tensor map) and not (row copies), one tile and several,
# volumes thinner than the filter
SHAPES = [(9, 17, 64), (20, 33, 136), (13, 16, 65), (5, 40, 131), (3, 2, 8), (1, 1, 1), (70, 18, 24)]


def codes(seed, shape, sfmt):
    r = np.random.RandomState(seed)
    q = r.randint(0, 256 if sfmt == synth.U8 else 65536, shape)
    return q.astype(np.uint8 if sfmt == synth.U8 else np.uint16)


def binomial(k):
    g = np.array([1.0])
    for _ in range(k - 1):
        g = np.convolve(g, [0.5, 0.5])
    return g.astype(np.float32)


def exact_codes(src, g, qs, qd):
    """Half-even codes of a filter whose weights are multiples of 2^-24: every sum is exact in
    64 bits, so exact ties are ties here too."""
    r = (len(g) - 1) // 2
    v = src.astype(np.float64)
    for ax in range(3):
        p = np.pad(v, [(r, r) if a == ax else (0, 0) for a in range(3)], mode="edge")
        n = v.shape[ax]
        v = sum(float(w) * np.take(p, range(i, i + n), axis=ax) for i, w in enumerate(g))
    return np.clip(np.rint(v * (qd / qs)), 0, qd)


def run(src, filt, dfmt, roi=None, offset=0):
    flat = torch.empty(src.size + offset, dtype=DT[synth.U8 if src.dtype == np.uint8 else synth.U16])
    flat[offset:] = torch.from_numpy(src.reshape(-1))
    t = flat.cuda()[offset:].view(src.shape)
    out = torch.zeros(src.shape, dtype=DT[dfmt], device="cuda")
    vkt.filter_tensor(t, filt, out=out, path="separable", roi=roi)
    torch.cuda.synchronize()
    vkt.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("k", [3, 5, 7, 9])
@pytest.mark.parametrize("offset", [0, 1])
def test_ties_round_to_even(shape, k, offset):
    """Binomial weights: a large share of the results are exact rounding ties.  offset 1: the
    source is not 16-byte aligned (plain loads)."""
    g = binomial(k)
    src = codes(k + sum(shape), shape, synth.U16)
    src[0] = 65535 if shape[0] % 2 else 0
    got = run(src, vkt.Filter.separable(g, g, g), synth.U16, offset=offset)
    np.testing.assert_array_equal(got.astype(np.float64), exact_codes(src, g, 65535.0, 65535.0))


@pytest.mark.parametrize("sfmt,dfmt", [(synth.U16, synth.U16), (synth.U8, synth.U16), (synth.U16, synth.U8)])
@pytest.mark.parametrize("k", [3, 5, 7])
def test_gaussian_codes_match_oracle(sfmt, dfmt, k):
    """Codes equal the 64-bit evaluation's wherever that is not within 1e-3 of a tie."""
    for shape in SHAPES:
        src = codes(3 * k + sum(shape), shape, sfmt)
        got = run(src, vkt.Filter.gaussian(k, 0.3 * k), dfmt)
        qd = 255.0 if dfmt == synth.U8 else 65535.0
        v = oracle.correlate(src, oracle.gaussian_weights(k, float(np.float32(0.3 * k))), 0.0, 1.0) * qd
        clear = np.abs(v - np.floor(v) - 0.5) > 1e-3
        np.testing.assert_array_equal(got[clear], np.clip(np.rint(v), 0, qd)[clear])


@pytest.mark.parametrize("roi", [((3, 2, 1), (70, 30, 17)), ((64, 16, 0), (65, 17, 20)), ((0, 0, 0), (136, 33, 20))])
def test_region_equals_whole_volume(roi):
    shape = (20, 33, 136)
    src = codes(5, shape, synth.U16)
    f = vkt.Filter.gaussian(5, 1.5)
    whole, part = run(src, f, synth.U16), run(src, f, synth.U16, roi=roi)
    (x0, y0, z0), (x1, y1, z1) = roi
    want = np.zeros_like(whole)
    want[z0:z1, y0:y1, x0:x1] = whole[z0:z1, y0:y1, x0:x1]
    np.testing.assert_array_equal(part, want)
