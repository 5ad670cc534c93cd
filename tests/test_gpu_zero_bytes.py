"""Bytes are scaled by a table or by a division that keeps zero off its slow path: slices with zero regions, with
every byte value, and of zeros alone match the oracle at each precision's bar."""
import numpy as np
import pytest

import oracle
import synth
from _common import TOL, infer, make_net, teacher_params

pytestmark = pytest.mark.gpu


def slices():
    rng = np.random.default_rng(8600)
    v = rng.integers(0, 256, size=(3, 64, 136), dtype=np.uint8)
    v[0].reshape(-1)[:512] = np.arange(512) % 256
    v[1, :, 40:100] = 0
    v[2] = 0
    return v


@pytest.mark.parametrize("name,prec", [("TEACHER", "bf16"), ("TEACHER", "fp32"), ("FASTMEMB", "bf16"), ("FASTMEMB", "fp32"),
                                       ("STUDENT", "fp32")])
def test_zero_bytes_match_oracle(name, prec):
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    layers = getattr(synth, name)
    seed = {"FASTMEMB": synth.FASTMEMB_WEIGHT_SEED, "STUDENT": synth.STUDENT_WEIGHT_SEED}.get(name)
    params = teacher_params() if name == "TEACHER" else synth.init_params(layers, seed)
    net = make_net(layers, {"bf16": m.MB_PREC_BF16, "fp32": m.MB_PREC_FP32}[prec], params)
    v = slices()
    out = infer(net, v)
    for i in range(3):
        err = np.abs(out[i] - oracle.forward_region(layers, params, v[i]))
        assert err.max() <= (1e-5 if prec == "fp32" else TOL["bf16"]["max_abs"]), (i, err.max())
    net.close()
