"""Dependent launches of the student nets and of FP16 MaskExtend: calls queued without a host
synchronisation between them share the net's workspace and follow one another's output, and give exactly
what calls on their own give. Through the C ABI."""
import numpy as np
import pytest

import synth
from _common import infer, make_net, student_params, teacher_params

pytestmark = pytest.mark.gpu


def lib():
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    return m


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_queued_student_calls_equal_single_calls(prec):
    import torch
    m = lib()
    code = {"fp32": m.MB_PREC_FP32, "bf16": m.MB_PREC_BF16}[prec]
    nets = [make_net(synth.STUDENT, code, student_params()) for _ in range(2)]
    shape = (2, 70, 300)
    vols = [synth.em_volume(8200 + i, *shape) for i in range(3)]
    want = [infer(nets[0], v) for v in vols]
    xs = [torch.from_numpy(v).cuda() for v in vols]
    streams = [torch.cuda.Stream() for _ in nets]
    outs = [[torch.empty(shape, device="cuda") for _ in range(6)] for _ in nets]
    torch.cuda.synchronize()
    for i in range(6):
        for net, st, out in zip(nets, streams, outs):
            m.mb_infer_volume(net.handle, xs[i % 3], *shape, out[i], stream=st)
    torch.cuda.synchronize()
    for out in outs:
        for i in range(6):
            np.testing.assert_array_equal(out[i].cpu().numpy(), want[i % 3])
    for n in nets:
        n.close()


def test_queued_mask_extend_calls_equal_single_calls():
    import torch
    m = lib()
    params = synth.init_params(synth.MASKEXTEND, 77, bias_std=0.01)
    nets = [make_net(synth.MASKEXTEND, m.MB_PREC_FP16, params) for _ in range(2)]
    z, h, w, steps = 7, 60, 200, 3
    em = torch.from_numpy(synth.em_volume(8300, z, h, w)).cuda()
    memb = 1.0 - em.float() / 255.0
    seeds = [(torch.rand((4, h, w), device="cuda") < p).to(torch.uint8).contiguous() for p in (0.2, 0.7)]

    def call(net, seed, masks, probs, st=None):
        m.mb_mask_extend_dir(net.handle, em, memb, z, h, w, seed, 2, steps, 1, masks, probs, stream=st)

    def buffers():
        return (torch.empty((steps, h, w), dtype=torch.uint8, device="cuda"),
                torch.empty((steps, 3, h, w), device="cuda"))

    want = []
    for seed in seeds:
        b = buffers()
        call(nets[0], seed, *b)
        torch.cuda.synchronize()
        want.append(b)
    streams = [torch.cuda.Stream() for _ in nets]
    got = [[buffers() for _ in range(4)] for _ in nets]
    torch.cuda.synchronize()
    for i in range(4):
        for net, st, out in zip(nets, streams, got):
            call(net, seeds[i % 2], *out[i], st)
    torch.cuda.synchronize()
    for out in got:
        for i in range(4):
            for a, b in zip(out[i], want[i % 2]):
                assert torch.equal(a, b)
    for n in nets:
        n.close()


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_training_after_its_targets_and_before_inference(prec):
    """The FP32 teacher writes the targets, the student takes its gradient, trains and maps, on one stream."""
    import torch
    m = lib()
    code = {"fp32": m.MB_PREC_FP32, "bf16": m.MB_PREC_BF16}[prec]
    teacher, net = make_net(synth.TEACHER, m.MB_PREC_FP32, teacher_params()), make_net(synth.STUDENT, code, student_params())
    z, h, w = 4, 60, 210
    vols = [synth.em_volume(8400 + i, z, h, w) for i in range(2)]
    x = [torch.from_numpy(v).cuda() for v in vols]
    t = [torch.from_numpy(infer(teacher, v)).cuda() for v in vols]
    ref = make_net(synth.STUDENT, code, student_params())
    want_grad, got_grad = (torch.empty(net.n_params, device="cuda") for _ in range(2))
    target, out = torch.zeros((z, h, w), device="cuda"), torch.empty((z, h, w), device="cuda")
    for i in (0, 1, 0):  # the targets of the call before are still in the buffer
        want = m.mb_student_loss_grad(ref.handle, x[i], t[i], z, h, w, want_grad)
        m.mb_infer_volume(teacher.handle, x[i], z, h, w, target)
        assert m.mb_student_loss_grad(net.handle, x[i], target, z, h, w, got_grad) == want
        assert torch.equal(got_grad, want_grad)
    cfg = m.train_cfg(batch=2, steps=3, seed=4)
    m.mb_student_train(ref.handle, x[1], t[1], z, h, w, cfg)
    m.mb_infer_volume(teacher.handle, x[1], z, h, w, target)
    m.mb_student_train(net.handle, x[1], target, z, h, w, cfg)
    m.mb_infer_volume(net.handle, x[0], z, h, w, out)
    a, b = (np.empty(net.n_params, np.float32) for _ in range(2))
    m.mb_get_weights(net.handle, a)
    m.mb_get_weights(ref.handle, b)
    np.testing.assert_array_equal(a, b)
    fresh = make_net(synth.STUDENT, code, a)
    np.testing.assert_array_equal(out.cpu().numpy(), infer(fresh, vols[0]))
    for n in (teacher, net, ref, fresh):
        n.close()


def test_fp32_student_in_several_chunks_equals_single_slices():
    """Three 4096 x 4096 slices pass the 3 GB of workspace that one chunk may take (two slices): the second
    chunk's first launch, a dependent one, overwrites the features that the first chunk's last one reads."""
    import torch
    m = lib()
    net = make_net(synth.STUDENT, m.MB_PREC_FP32, student_params())
    z, h, w = 3, 4096, 4096
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    x = torch.randint(0, 256, (z, h, w), dtype=torch.uint8, device="cuda", generator=g)
    out, one = torch.empty((z, h, w), device="cuda"), torch.empty((1, h, w), device="cuda")
    before = m.launch_count()
    m.mb_infer_volume(net.handle, x, z, h, w, out)
    assert m.launch_count() - before == 4
    for i in range(z):
        m.mb_infer_volume(net.handle, x[i], 1, h, w, one)
        torch.cuda.synchronize()
        assert torch.equal(out[i], one[0])
    net.close()
