"""FP32 student inference on the tensor cores (three-part BF16 split) against the CUDA-core kernels and the
oracle. The net scaled by 2^40 (first layer) and 2^-40 (second layer's weights) is the same network exactly
but beyond the split's range, so it runs on the CUDA cores.

Tolerance: both paths sum 9 and 144 products per output; an FP32 chain's relative error is below 1e-6 a
layer on a logit of order 1, which the sigmoid's slope of at most 1/4 scales: 2e-6 on a probability for
the two together is generous. Against the oracle the split path may not be worse than the CUDA cores by
more than one rounding of a probability (6e-8)."""
import numpy as np
import pytest

import oracle
import synth
from _common import infer, make_net

pytestmark = pytest.mark.gpu

SCALE = np.float32(2.0 ** 40)


def params():
    return synth.init_params(synth.STUDENT, synth.STUDENT_WEIGHT_SEED, bias_std=0.05)


@pytest.fixture(scope="module")
def nets():
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    q = params()
    q[:160] *= SCALE
    q[160:2464] /= SCALE
    a, b = make_net(synth.STUDENT, m.MB_PREC_FP32, params()), make_net(synth.STUDENT, m.MB_PREC_FP32, q)
    yield a, b
    a.close()
    b.close()


@pytest.mark.parametrize("shape", [(1, 8, 8), (3, 17, 15), (1, 33, 126), (2, 9, 127), (1, 20, 128), (1, 12, 129), (1, 8, 385),
                                   (1, 300, 31)])
def test_split_inference_equals_cuda_cores(nets, shape):
    v = synth.em_volume(8300 + shape[2], *shape)
    got, ref = (infer(n, v) for n in nets)
    assert np.abs(got - ref).max() <= 2e-6
    exact = oracle.forward_region(synth.STUDENT, params(), v[0])
    assert np.abs(got[0] - exact).max() <= np.abs(ref[0] - exact).max() + 6e-8
    q = infer(nets[0], v, 1)
    np.testing.assert_array_equal(q, np.minimum(255, np.floor(np.float32(255.0) * got + np.float32(0.5))).astype(np.uint8))


@pytest.mark.parametrize("rows,cols", [(1, 1), (2, 127), (3, 128), (5, 129), (61, 257), (96, 300)])
def test_region_equals_crop(nets, rows, cols):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    H, W = 96, 300
    v = synth.em_volume(8400, 2, H, W)
    full = infer(nets[0], v)
    x = torch.from_numpy(v).cuda()
    for y0, x0 in ((0, 0), (H - rows, W - cols), ((H - rows) // 2, (W - cols) // 2)):
        out = torch.full((2 * rows * cols + cols,), 7.0, dtype=torch.float32, device="cuda")
        m.mb_infer_region(nets[0].handle, x, 2, H, W, y0, x0, rows, cols, out)
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        np.testing.assert_array_equal(got[:2 * rows * cols].reshape(2, rows, cols), full[:, y0:y0 + rows, x0:x0 + cols])
        assert (got[2 * rows * cols:] == 7.0).all()


def test_timed_out_wait_is_reported(nets, monkeypatch):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    lib = m.load()
    v = synth.em_volume(8500, 1, 40, 50)
    ref = infer(nets[0], v)
    x = torch.from_numpy(v).cuda()
    out = torch.zeros((1, 40, 50), dtype=torch.float32, device="cuda")
    call = lambda: lib.mb_infer_volume(nets[0].handle, x.data_ptr(), 1, 40, 50, out.data_ptr(), 0, None)
    monkeypatch.setenv("MB_FAULT_STALL", "1")
    assert call() == m.MB_OK
    torch.cuda.synchronize()
    monkeypatch.delenv("MB_FAULT_STALL")
    assert call() == m.MB_ERR_TIMEOUT
    assert call() == m.MB_OK
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), ref)
