"""Failure detection in the kernels that answer by size, format and filter (test_fault_gpu.py has the
general direct kernel): the load of every CTA's first plane is withheld, the bounded waits run out,
nothing is written, the timeout is reported, and the next call is right again."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2203_10213_gb300 as vkt  # noqa: E402

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

GAUSS3, GAUSS5 = vkt.Filter.gaussian(3, 1.0), vkt.Filter.gaussian(5, 1.5)
CROSS = np.zeros((3, 3, 3), np.float32)
CROSS[1, 1, :] = CROSS[1, :, 1] = CROSS[:, 1, 1] = 0.125
STAR = vkt.Filter.dense(CROSS)
DENSE3 = vkt.Filter.dense(np.random.RandomState(1).standard_normal((3, 3, 3)).astype(np.float32))

# what the log calls the kernel, (nz, ny, nx), source, destination, filter, path.  The split brick takes
# three planes (no vote of its warps before the last plane) and many.
CASES = [
    ("separable-split", (3, 33, 136), torch.uint16, torch.uint16, GAUSS5, "separable"),
    ("separable-split", (70, 33, 136), torch.uint16, torch.uint16, GAUSS5, "separable"),
    ("separable-split", (20, 18, 64), torch.uint8, torch.uint16, GAUSS5, "separable"),
    ("direct-star", (24, 32, 48), torch.uint8, torch.float32, STAR, "direct"),
    ("direct-star", (3, 33, 136), torch.uint16, torch.float32, STAR, "direct"),
    ("direct-march", (64, 1216, 128), torch.float32, torch.float32, DENSE3, "direct"),
    ("separable-walk", (64, 1216, 128), torch.uint8, torch.float32, GAUSS3, "separable"),
    ("separable-walk", (1, 33, 136), torch.float32, torch.float32, GAUSS3, "separable"),
    ("separable-walk", (30, 17, 64), torch.float32, torch.float32, GAUSS5, "separable"),
]


def source(shape, dtype):
    r = np.random.RandomState(3)
    if dtype == torch.float32:
        return torch.from_numpy(r.standard_normal(shape).astype(np.float32)).cuda()
    wide = dtype == torch.uint16
    return torch.from_numpy(r.randint(0, 65536 if wide else 256, shape).astype(np.uint16 if wide else np.uint8)).cuda()


@pytest.mark.parametrize("case", range(len(CASES)))
def test_withheld_load_is_reported(case, capfd):
    mark, shape, sdt, ddt, filt, path = CASES[case]
    src = source(shape, sdt)
    out = torch.zeros(shape, dtype=ddt, device="cuda")
    want = vkt.filter_tensor(src, filt, out=torch.zeros_like(out), path=path)
    vkt.synchronize()
    capfd.readouterr()
    with vkt.policy(debug=vkt.DEBUG_INJECT_WAIT_TIMEOUT | vkt.DEBUG_LOG):
        vkt.filter_tensor(src, filt, out=out, path=path)
        t0 = time.monotonic()
        code = vkt._lib.vktSynchronize()
        waited = time.monotonic() - t0
    assert mark in capfd.readouterr().err
    assert vkt.ERRORS.get(code) == "VKT_ERROR_DEVICE_TIMEOUT", code
    assert 1.0 < waited < 20.0, waited
    assert not out.cpu().numpy().any()          # no CTA wrote
    assert vkt._lib.vktSynchronize() == 0       # the status was cleared
    vkt.filter_tensor(src, filt, out=out, path=path)
    vkt.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), want.cpu().numpy())
