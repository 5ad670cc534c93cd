"""A training run whose device-side wait runs out (the producers withhold their arrivals: a flag that the
host sets) reports MB_ERR_TIMEOUT and keeps nothing of the run: the checkpoint file, the net's weights and
the loss curve are those of before the call, and training goes on from there as if the call had not been
made. Through the C ABI."""
import ctypes

import numpy as np
import pytest

import synth
from _common import infer, make_net, student_params

pytestmark = pytest.mark.gpu

Z, H, W = 6, 48, 150


def data():
    v = synth.em_volume(7700, Z, H, W)
    return v, (1.0 / (1.0 + np.exp((v.astype(np.float32) - 120.0) / 20.0))).astype(np.float32)


def train(net, steps, ckpt=None, resume=0):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    v, t = data()
    curve = np.full(steps, -1.0, np.float32)
    cfg = m.train_cfg(batch=2, steps=steps, ckpt_every=2, resume=resume, seed=3)
    status = m.load().mb_student_train(net.handle, torch.from_numpy(v).cuda().data_ptr(),
                                       torch.from_numpy(t).cuda().data_ptr(), Z, H, W, ctypes.byref(cfg),
                                       str(ckpt).encode() if ckpt else None, curve.ctypes.data, None)
    message = m.last_error()
    weights = np.empty(net.n_params, np.float32)
    m.mb_get_weights(net.handle, weights)
    return status, weights, curve, message


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("resume", [0, 1])
def test_timed_out_training_keeps_nothing(prec, resume, tmp_path, monkeypatch):
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    code = {"fp32": m.MB_PREC_FP32, "bf16": m.MB_PREC_BF16}[prec]
    v = data()[0][:1]
    whole = make_net(synth.STUDENT, code, student_params())
    assert train(whole, 6)[0] == m.MB_OK
    net, ckpt = make_net(synth.STUDENT, code, student_params()), tmp_path / "student.ckpt"
    status, before, _, _ = train(net, 4, ckpt)
    assert status == m.MB_OK
    blob, map_before = ckpt.read_bytes(), infer(net, v)
    monkeypatch.setenv("MB_FAULT_STALL", "1")
    status, after, curve, message = train(net, 6, ckpt, resume)
    monkeypatch.delenv("MB_FAULT_STALL")
    assert status == m.MB_ERR_TIMEOUT and "training" in message and "wait limit" in message
    assert ckpt.read_bytes() == blob
    np.testing.assert_array_equal(after, before)
    assert (curve == -1.0).all()
    np.testing.assert_array_equal(infer(net, v), map_before)
    status, resumed, _, _ = train(net, 6, ckpt, 1)
    assert status == m.MB_OK
    want = np.empty(whole.n_params, np.float32)
    m.mb_get_weights(whole.handle, want)
    np.testing.assert_array_equal(resumed, want)
    net.close()
    whole.close()


def test_inference_that_timed_out_does_not_fail_a_training_run(monkeypatch):
    import torch
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    net, lib = make_net(synth.STUDENT, m.MB_PREC_FP32, student_params()), m.load()
    x = torch.from_numpy(data()[0]).cuda()
    out = torch.empty((Z, H, W), device="cuda")
    call = (net.handle, x.data_ptr(), Z, H, W, out.data_ptr(), 0, None)
    monkeypatch.setenv("MB_FAULT_STALL", "1")
    assert lib.mb_infer_volume(*call) == m.MB_OK
    torch.cuda.synchronize()
    monkeypatch.delenv("MB_FAULT_STALL")
    assert train(net, 2)[0] == m.MB_OK
    assert lib.mb_infer_volume(*call) == m.MB_ERR_TIMEOUT
    assert "training" not in m.last_error() and "wait limit" in m.last_error()
    assert lib.mb_infer_volume(*call) == m.MB_OK
    torch.cuda.synchronize()
    net.close()
