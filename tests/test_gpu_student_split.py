"""The student's training passes on the tensor cores (three-part BF16 split) against the CUDA-core passes
that run where the weights leave the split's range. A net whose first layer is scaled by 2^40 and whose
second layer's weights by 2^-40 is the same network exactly (powers of two commute with ReLU), but
its weights are beyond the bound, so it trains on the CUDA cores; its gradients are those of the plain
net times 2^-40 (first layer) and 2^40 (second layer's weights), also exactly.

Tolerance: the oracle test holds either path's gradient to 1e-4 of its largest element; the two paths
are held to the same of one another, element by element of each of the four parts (an FP32 chain of 144
products has a relative error below 1e-5, and sums over pixels cancel by about an order of magnitude)."""
import numpy as np
import pytest

import synth
from _common import make_net

pytestmark = pytest.mark.gpu

PARTS = {"W1": slice(0, 144), "b1": slice(144, 160), "W2": slice(160, 2464), "rest": slice(2464, None)}
SCALE = np.float32(2.0 ** 40)


@pytest.fixture(scope="module")
def nets():
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    p = synth.init_params(synth.STUDENT, synth.STUDENT_WEIGHT_SEED, bias_std=0.05)
    q = p.copy()
    q[:160] *= SCALE
    q[PARTS["W2"]] /= SCALE
    a, b = make_net(synth.STUDENT, m.MB_PREC_FP32, p), make_net(synth.STUDENT, m.MB_PREC_FP32, q)
    yield a, b
    a.close()
    b.close()


def loss_grad(net, v, tgt):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    g = torch.empty(net.n_params, dtype=torch.float32, device="cuda")
    loss = m.mb_student_loss_grad(net.handle, torch.from_numpy(v).cuda(), torch.from_numpy(tgt).cuda(), *v.shape, g)
    return loss, g.cpu().numpy()


# strips of 128 columns (with two more for the first layer's gradient), tiles of 16 x 16, few and many rows
@pytest.mark.parametrize("shape", [(1, 8, 8), (3, 16, 16), (2, 17, 15), (1, 33, 126), (1, 20, 127), (1, 9, 128),
                                   (2, 12, 129), (1, 300, 31), (1, 8, 385)])
def test_split_gradient_equals_cuda_cores(nets, shape):
    v = synth.em_volume(7800 + shape[2], *shape)
    tgt = np.random.default_rng(shape[2]).uniform(0.05, 0.95, size=shape).astype(np.float32)
    (la, ga), (lb, gb) = (loss_grad(n, v, tgt) for n in nets)
    assert abs(la - lb) <= 1e-5 * abs(lb)
    gb[:160] *= SCALE
    gb[PARTS["W2"]] /= SCALE
    for name, s in PARTS.items():
        assert np.abs(ga[s] - gb[s]).max() <= 1e-4 * np.abs(gb[s]).max(), name


def test_stalled_split_pass_times_out(nets, monkeypatch):
    from paper_1612_02120_gb300 import membrane as m
    v = synth.em_volume(7900, 1, 40, 40)
    tgt = np.full(v.shape, 0.5, dtype=np.float32)
    loss, g = loss_grad(nets[0], v, tgt)
    monkeypatch.setenv("MB_FAULT_STALL", "1")
    with pytest.raises(m.MembraneError, match="wait limit"):
        loss_grad(nets[0], v, tgt)
    monkeypatch.delenv("MB_FAULT_STALL")
    again, h = loss_grad(nets[0], v, tgt)
    assert again == loss
    np.testing.assert_array_equal(h, g)
