"""The FP32 layers on the tensor cores (three-part BF16 split) against the CUDA-core kernels they replace
and against the oracle. A net whose first layer is scaled by 2^104 and whose second layer by 2^-104 is
the same network exactly (powers of two commute with ReLU, max-out and max-filters), but its activations
are beyond the range that the split path accepts, so it runs on the CUDA cores.

Tolerance: both paths sum at most 800 products per output and layer; an FP32 FMA chain's relative error
is below 1e-6 and each of the 3 to 5 layers adds its own to a logit of order 1, which the sigmoid's slope
of at most 1/4 scales: 2e-6 on a probability (the teacher and FastMemb; FastMemb_3nm's zero-mean head
cancels, so that net is held to the oracle alone). Against the oracle the split path may not be worse than
the FMA path by more than one rounding of a probability (6e-8)."""
import numpy as np
import pytest

import oracle
import synth
from _common import infer, make_net, teacher_params

pytestmark = pytest.mark.gpu

BIG = np.float32(2.0 ** 104)
TOL = 2e-6


def scaled(params, n1, n2):
    """First layer (n1 parameters, W and b) times 2^104, the second layer's n2 weights times 2^-104."""
    p = params.copy()
    p[:n1] *= BIG
    p[n1:n1 + n2] /= BIG
    assert np.isfinite(p).all()
    return p


def pair(layers, params, n1, n2):
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    return make_net(layers, m.MB_PREC_FP32, params), make_net(layers, m.MB_PREC_FP32, scaled(params, n1, n2))


@pytest.fixture(scope="module")
def teacher():
    a, b = pair(synth.TEACHER, teacher_params(), 832, 25600)
    yield a, b
    a.close()
    b.close()


@pytest.mark.parametrize("shape", [(1, 8, 8), (2, 9, 118), (1, 130, 123), (3, 17, 124), (1, 70, 128), (1, 40, 251),
                                   (2, 33, 257)])
def test_teacher_split_path_equals_cuda_cores(teacher, shape):
    v = synth.em_volume(7300 + shape[2], *shape)
    got, ref = (infer(n, v) for n in teacher)
    assert np.abs(got - ref).max() <= TOL
    if shape[1] <= 40:
        exact = oracle.forward_region(synth.TEACHER, teacher_params(), v[0])
        assert np.abs(got[0] - exact).max() <= np.abs(ref[0] - exact).max() + 6e-8
    q = infer(teacher[0], v, 1)
    assert np.array_equal(q, np.minimum(255, np.floor(np.float32(255.0) * got + np.float32(0.5))).astype(np.uint8))


@pytest.mark.parametrize("name", ["fastmemb", "fastmemb_3nm"])
def test_fastmemb_split_path_equals_cuda_cores(name):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    layers, params = {"fastmemb": (synth.FASTMEMB, synth.init_params(synth.FASTMEMB, synth.FASTMEMB_WEIGHT_SEED)),
                      "fastmemb_3nm": (synth.FASTMEMB_3NM, synth.init_params(
                          synth.FASTMEMB_3NM, synth.FASTMEMB_3NM_WEIGHT_SEED, center_head=True))}[name]
    a, b = pair(layers, params, 64 * 16 + 64, 64 * 32 * 16)
    for shape in ((1, 55, 57), (2, 61, 129), (1, 150, 213)):
        v = synth.em_volume(7400 + shape[2], *shape)
        got, ref = infer(a, v), infer(b, v)
        if name == "fastmemb":
            assert np.abs(got - ref).max() <= TOL, shape
        exact = oracle.forward_region(layers, params, v[0])
        assert np.abs(got[0] - exact).max() <= np.abs(ref[0] - exact).max() + 6e-8, shape
        x = torch.from_numpy(v).cuda()
        sub = torch.empty((shape[0], (shape[1] + 1) // 2, (shape[2] + 1) // 2), device="cuda")
        m.mb_infer_volume_subsampled(a.handle, x, *shape, 2, sub)
        torch.cuda.synchronize()
        assert np.array_equal(sub.cpu().numpy(), got[:, ::2, ::2])
    a.close()
    b.close()


def test_timed_out_wait_is_reported(teacher, monkeypatch):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    net = teacher[0]
    v = synth.em_volume(7500, 1, 32, 40)
    want = infer(net, v)
    x = torch.from_numpy(v).cuda()
    out = torch.empty((1, 32, 40), device="cuda")
    lib = m.load()
    monkeypatch.setenv("MB_FAULT_STALL", "1")
    assert lib.mb_infer_volume(net.handle, x.data_ptr(), 1, 32, 40, out.data_ptr(), 0, None) == m.MB_OK
    torch.cuda.synchronize()
    monkeypatch.delenv("MB_FAULT_STALL")
    assert lib.mb_infer_volume(net.handle, x.data_ptr(), 1, 32, 40, out.data_ptr(), 0, None) == m.MB_ERR_TIMEOUT
    assert "wait limit" in m.last_error()
    assert np.array_equal(infer(net, v), want)
