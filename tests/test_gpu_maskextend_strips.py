"""MaskExtend FP16 at the edges of its strips (128 conv columns, of which the layers' dilated max-filters
keep 127, 126, 124 and 120) and of its row groups, in both directions: one step against the FP32 path
within the 16-bit bar (the FP32 path is held to the oracle in its own tests; the bar is the oracle's)."""
import numpy as np
import pytest

import synth
from _common import TOL, make_net

pytestmark = pytest.mark.gpu

M = synth.MASKEXTEND


@pytest.fixture(scope="module")
def nets():
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    p = synth.init_params(M, synth.MASKEXTEND_WEIGHT_SEED)
    pair = make_net(M, m.MB_PREC_FP16, p), make_net(M, m.MB_PREC_FP32, p)
    yield pair
    for n in pair:
        n.close()


@pytest.mark.parametrize("direction", [1, -1])
@pytest.mark.parametrize("shape", [(55, 120), (56, 121), (57, 124), (63, 125), (64, 126), (65, 127), (66, 128), (67, 129),
                                   (129, 55), (120, 256), (71, 257)])
def test_one_step_equals_fp32_path(nets, shape, direction):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    h, w = shape
    em = synth.em_volume(9600 + w, 8, h, w)
    memb = synth.membrane_maps(em)
    seeds = synth.disk_masks(4, h, w, h / 2, w / 2, min(h, w) / 4, 1.0, -0.5)
    d_em, d_memb, d_seeds = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (em, memb, seeds))
    probs = []
    for net in nets:
        masks = torch.zeros((1, h, w), dtype=torch.uint8, device="cuda")
        pr = torch.full((1, 3, h, w), -1.0, dtype=torch.float32, device="cuda")
        m.mb_mask_extend_dir(net.handle, d_em, d_memb, 8, h, w, d_seeds, 4, 1, direction, masks, pr)
        torch.cuda.synchronize()
        probs.append(pr.cpu().numpy())
    err = np.abs(probs[0] - probs[1])
    assert err.max() <= TOL["fp16"]["max_abs"] and err.mean() <= TOL["fp16"]["mean_abs"]
