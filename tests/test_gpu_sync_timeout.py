"""Calls that synchronise return MB_OK only for complete maps: where a device-side wait ran out (the
kernels' producers withhold their arrivals: a flag that the host sets), the call itself says so, for every
net family, and the next call is right again. Through the C ABI."""
import ctypes

import numpy as np
import pytest

import synth
from _common import infer, make_net, student_params, teacher_params

pytestmark = pytest.mark.gpu

Z, H, W = 2, 64, 130
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


def net_of(name):
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    layers, prec, params = NETS[name]
    return make_net(layers, getattr(m, prec), params())


@pytest.mark.parametrize("mode", ["MB_HOST_IO_AUTO", "MB_HOST_IO_SLABS"])
@pytest.mark.parametrize("name", list(NETS))
def test_host_volume_reports_a_timed_out_wait(name, mode, monkeypatch):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    net, lib = net_of(name), m.load()
    m.mb_set_host_io(net.handle, getattr(m, mode))
    v = synth.em_volume(7800, Z, H, W)
    want = infer(net, v)
    x, out = torch.from_numpy(v).pin_memory(), torch.full((Z, H, W), -1.0).pin_memory()
    call = (net.handle, x.data_ptr(), Z, H, W, out.data_ptr(), 0, None)
    monkeypatch.setenv("MB_FAULT_STALL", "1")
    assert lib.mb_infer_volume(*call) == m.MB_ERR_TIMEOUT
    assert "wait limit" in m.last_error() and "training" not in m.last_error()
    monkeypatch.delenv("MB_FAULT_STALL")
    assert lib.mb_infer_volume(*call) == m.MB_OK
    np.testing.assert_array_equal(out.numpy(), want)
    net.close()


@pytest.mark.parametrize("student", ["student_fp32", "student_bf16"])
@pytest.mark.parametrize("teacher", ["teacher_fp32", "teacher_bf16"])
@pytest.mark.parametrize("max_frac", [0.0, 1.0])  # every tile recomputed by the teacher, or none
def test_cascade_reports_a_timed_out_wait(student, teacher, max_frac, monkeypatch):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    s, t, lib = net_of(student), net_of(teacher), m.load()
    v = synth.em_volume(7800, Z, H, W)
    want = infer(t if max_frac == 0.0 else s, v)
    x, out, rate = torch.from_numpy(v).cuda(), torch.full((Z, H, W), -1.0, device="cuda"), ctypes.c_double()
    call = (s.handle, t.handle, x.data_ptr(), Z, H, W, out.data_ptr(), 32, 0.0, 1.0, max_frac, ctypes.byref(rate),
            None, None)
    assert lib.mb_infer_cascade(*call) == m.MB_OK
    monkeypatch.setenv("MB_FAULT_STALL", "1")
    assert lib.mb_infer_cascade(*call) == m.MB_ERR_TIMEOUT
    assert "wait limit" in m.last_error()
    monkeypatch.delenv("MB_FAULT_STALL")
    assert lib.mb_infer_cascade(*call) == m.MB_OK
    assert rate.value == (1.0 if max_frac == 0.0 else 0.0)
    np.testing.assert_array_equal(out.cpu().numpy(), want)
    s.close()
    t.close()
