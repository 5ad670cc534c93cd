"""The 16-bit FastMemb layers at the edges of their strips and items: a region's map does not depend on
where the strips and the CTAs' row ranges fall, so regions of awkward sizes and odd origins equal the
crop of the whole slice's map bitwise (the whole map is held to the oracle in test_gpu_fastmemb.py)."""
import numpy as np
import pytest

import synth
from _common import infer, make_net

pytestmark = pytest.mark.gpu

NETS = {"fastmemb": (synth.FASTMEMB, synth.FASTMEMB_WEIGHT_SEED, False),
        "fastmemb_3nm": (synth.FASTMEMB_3NM, synth.FASTMEMB_3NM_WEIGHT_SEED, True)}


@pytest.mark.parametrize("name", list(NETS))
@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_regions_equal_the_whole_map_bitwise(name, prec):
    import torch
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    layers, seed, center = NETS[name]
    net = make_net(layers, {"bf16": m.MB_PREC_BF16, "fp16": m.MB_PREC_FP16}[prec],
                   synth.init_params(layers, seed, center_head=center))
    h, w = 301, 411
    v = synth.em_volume(7100, 2, h, w)
    whole = infer(net, v)
    x = torch.from_numpy(v).cuda()
    # widths at which a layer's last strip holds one column, is full, or is one over; short regions
    # leave most CTAs one or two rows of several columns
    for rows, cols in ((1, 1), (2, 3), (7, 102), (3, 103), (1, 127), (5, 128), (9, 129), (17, 250), (64, 33), (300, 410)):
        y0, x0 = (h - rows) // 2 | 1 if rows < 299 else 1, 1
        out = torch.full((2, rows, cols), -1.0, device="cuda")
        m.mb_infer_region(net.handle, x, 2, h, w, y0, x0, rows, cols, out)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), whole[:, y0:y0 + rows, x0:x0 + cols]), (rows, cols)
    sub = torch.empty((2, (h + 1) // 2, (w + 1) // 2), device="cuda")
    m.mb_infer_volume_subsampled(net.handle, x, 2, h, w, 2, sub)
    torch.cuda.synchronize()
    assert np.array_equal(sub.cpu().numpy(), whole[:, ::2, ::2])
    net.close()
