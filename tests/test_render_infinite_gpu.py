"""Rendering where a sample lies exactly on a voxel or a table entry and its neighbours are infinite:
the blend takes that voxel or entry with weight 1 and the one above it with weight 0, never the one
below it (0 times infinity is NaN, and a NaN value is classified as 0)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    import paper_2203_10213_gb300 as vkt

LUT = np.array([[0, 0, 0.2, 0.05], [0.2, 0.5, 0.8, 0.1], [0.5, 0.1, 0.3, 0.15], [1, 0.8, 0.4, 0.25]], np.float32)


def ray(v, lut):
    """The pixel of a ray along z through the middle column, one sample on every voxel."""
    nz, ny, nx = v.shape
    dims = tuple(float(n) for n in (nx, ny, nz))
    got = vkt.render(torch.from_numpy(v).cuda(), 1, 1, (dims[0] / 2, dims[1] / 2, -8.0),
                     (dims[0] / 2, dims[1] / 2, dims[2] / 2), (0.0, 1.0, 0.0), 0.5, 1.0, lut)
    vkt.synchronize()
    return got.cpu().numpy()[0, 0]


def reference(v, lut):
    """The same in 64 bits; every voxel of the cell is multiplied by its weight, zeros too."""
    nz, ny, nx = v.shape
    x, y = (nx - 1) // 2, (ny - 1) // 2
    out, opacity = np.zeros(3), 0.0
    with np.errstate(invalid="ignore"):
        for z in range(nz):
            c = v[min(z, nz - 1):z + 2, y:y + 2, x:x + 2].astype(np.float64)
            s = c[:, :, 0] * 1.0 + c[:, :, 1] * 0.0
            s = s[:, 0] * 1.0 + s[:, 1] * 0.0
            s = s[0] * 1.0 + s[1] * 0.0 if z + 1 < nz else s[0]
            u = 0.0 if np.isnan(s) else min(max(s, 0.0), 1.0)
            f = u * (len(lut) - 1)
            i = min(int(f), len(lut) - 2)
            e = lut[i].astype(np.float64) * (1.0 - (f - i)) + lut[i + 1].astype(np.float64) * (f - i)
            out += (1.0 - opacity) * e[3] * e[:3]
            opacity += (1.0 - opacity) * e[3]
    return np.append(out, opacity)


# the middle column at odd and even voxels, the infinite voxel beside it along each axis
@pytest.mark.parametrize("nx,ny", [(9, 9), (11, 11), (9, 11), (11, 9)])
@pytest.mark.parametrize("dx,dy,z", [(0, 0, 6), (0, 0, 7), (-1, 0, 4), (1, 0, 4), (0, -1, 9), (0, 1, 9),
                                     (-1, -1, 5), (1, 1, 12)])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_infinite_voxel(nx, ny, dx, dy, z, sign):
    v = np.random.RandomState(nx * 16 + ny).random_sample((16, ny, nx)).astype(np.float32)
    v[z, (ny - 1) // 2 + dy, (nx - 1) // 2 + dx] = sign * np.inf
    # 16 samples, each good to a few units of 2^-22; the classification of a sample as 0 or not
    # changes the pixel by 0.01 and more
    np.testing.assert_allclose(ray(v, LUT), reference(v, LUT), rtol=0, atol=5e-5)


# the values that classify exactly to entry i of four
@pytest.mark.parametrize("entry", range(4))
@pytest.mark.parametrize("infinite", range(4))
def test_infinite_entry(entry, infinite):
    lut = LUT.copy()
    lut[infinite, 0] = np.inf
    v = np.full((16, 9, 9), np.float32(entry) / np.float32(3), np.float32)
    got, ref = ray(v, lut), reference(v, lut)
    np.testing.assert_allclose(got[1:], ref[1:], rtol=0, atol=5e-5)
    i = min(entry, 2)          # the cell of entries i and i + 1
    if infinite not in (i, i + 1):
        assert np.isfinite(got[0])
    else:
        # infinite where that entry has weight 1, else NaN by 0 times infinity
        assert np.isposinf(got[0]) if infinite == entry else np.isnan(got[0])
