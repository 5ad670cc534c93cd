"""Host volumes whose slices hold an odd number of bytes: in slabs, the float maps follow the input bytes in a
device buffer and have to start on a boundary of their own. Every net family, both output types, several slabs
for the smallest net; bitwise the device path's maps. Through the C ABI."""
import numpy as np
import pytest

import synth
from _common import infer, make_net, student_params, teacher_params

pytestmark = pytest.mark.gpu

NETS = {
    "teacher_bf16": (synth.TEACHER, "MB_PREC_BF16", teacher_params),
    "teacher_fp32": (synth.TEACHER, "MB_PREC_FP32", teacher_params),
    "student_bf16": (synth.STUDENT, "MB_PREC_BF16", student_params),
    "student_fp32": (synth.STUDENT, "MB_PREC_FP32", student_params),
    "fastmemb_bf16": (synth.FASTMEMB, "MB_PREC_BF16",
                      lambda: synth.init_params(synth.FASTMEMB, synth.FASTMEMB_WEIGHT_SEED)),
    "fastmemb_fp32": (synth.FASTMEMB, "MB_PREC_FP32",
                      lambda: synth.init_params(synth.FASTMEMB, synth.FASTMEMB_WEIGHT_SEED)),
}
CASES = [(name, s) for name in NETS for s in ((1, 27, 29), (3, 31, 33), (2, 45, 27))] + [("student_bf16", (7, 1501, 1503))]


@pytest.mark.parametrize("name,shape", CASES)
@pytest.mark.parametrize("out_type", [0, 1])
def test_odd_slices_in_slabs_equal_the_device_path(name, shape, out_type):
    import torch
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    layers, prec, params = NETS[name]
    net = make_net(layers, getattr(m, prec), params())
    m.mb_set_host_io(net.handle, m.MB_HOST_IO_SLABS)
    v = np.random.default_rng(7).integers(0, 256, shape, dtype=np.uint8)
    want = infer(net, v, out_type)
    for pinned in (True, False):
        x, out = torch.from_numpy(v), torch.zeros(shape, dtype=torch.float32 if out_type == 0 else torch.uint8)
        if pinned:
            x, out = x.pin_memory(), out.pin_memory()
        m.mb_infer_volume(net.handle, x, *shape, out, out_type)
        np.testing.assert_array_equal(out.numpy(), want)
    net.close()
