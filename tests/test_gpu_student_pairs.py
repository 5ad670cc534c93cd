"""BF16 student inference hands rows over two at a time: an odd last row's partner is computed and
not stored, and a CTA's range may begin at any row pair. A pixel's value depends on neither, so a
region of any size equals the crop of the full map exactly, and nothing past its end is written."""
import numpy as np
import pytest

import synth
from _common import infer, make_net, student_params

pytestmark = pytest.mark.gpu

H, W = 163, 391


@pytest.fixture(scope="module")
def net_and_map():
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    n = make_net(synth.STUDENT, m.MB_PREC_BF16, student_params())
    v = synth.em_volume(7700, 2, H, W)
    yield n, v, infer(n, v)
    n.close()


@pytest.mark.parametrize("u8", [False, True])
@pytest.mark.parametrize("rows", [1, 2, 3, 7, 8, 9, H])
@pytest.mark.parametrize("cols", [1, 125, 126, 127, 253, W])
def test_region_of_any_size_equals_crop(net_and_map, rows, cols, u8):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    net, v, full = net_and_map
    x = torch.from_numpy(v).cuda()
    kind = m.MB_OUT_U8 if u8 else m.MB_OUT_F32
    want = np.minimum(255, np.floor(np.float32(255.0) * full + np.float32(0.5))).astype(np.uint8) if u8 else full
    for y0, x0 in ((0, 0), (H - rows, W - cols), ((H - rows) // 2, (W - cols) // 2)):
        buf = torch.full((2 * rows * cols + cols,), 7, dtype=torch.uint8 if u8 else torch.float32, device="cuda")
        m.mb_infer_region(net.handle, x, 2, H, W, y0, x0, rows, cols, buf, kind)
        torch.cuda.synchronize()
        got = buf.cpu().numpy()
        np.testing.assert_array_equal(got[:2 * rows * cols].reshape(2, rows, cols), want[:, y0:y0 + rows, x0:x0 + cols])
        assert (got[2 * rows * cols:] == 7).all()
