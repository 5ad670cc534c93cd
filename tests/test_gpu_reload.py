"""New weights in a net that has run before: every later call uses them, bitwise as a fresh net does. A
batch is captured into a graph that the library keeps for the same block list; loading weights or
calibrating again may not leave parts of the old ones in it. Through the C ABI."""
import numpy as np
import pytest

import synth
from _common import make_net, student_params, teacher_params

pytestmark = pytest.mark.gpu

T = synth.TEACHER
SHAPES = [(2, 37, 130), (1, 64, 40)]


def other_params(params, seed):
    """Other weights of the same scales (biases and the head's among them)."""
    rng = np.random.default_rng(seed)
    return (params * rng.uniform(0.5, 1.5, params.size)).astype(np.float32)


def batch_of(seed):
    import torch
    xs = [torch.from_numpy(synth.em_volume(seed + i, *s)).cuda() for i, s in enumerate(SHAPES)]
    outs = [torch.empty(s, device="cuda") for s in SHAPES]
    blocks = [(x, *s, s[2], s[1] * s[2], o, s[2], s[1] * s[2]) for x, o, s in zip(xs, outs, SHAPES)]
    return xs, outs, blocks


def run_batch(net, outs, blocks, per_block=False):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    for o in outs:
        o.fill_(-1.0)
    (m.mb_infer_batch_per_block if per_block else m.mb_infer_batch)(net.handle, blocks)
    torch.cuda.synchronize()
    return [o.cpu().numpy() for o in outs]


def calibrate(net, seed, gain=1):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    v = np.minimum(synth.em_volume(seed, 2, 64, 64).astype(np.int64) // gain, 255).astype(np.uint8)
    m.mb_calibrate_fp8(net.handle, torch.from_numpy(v).cuda(), 2, 64, 64)


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
def test_batch_after_a_reload_uses_the_new_weights(prec):
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    code = {"bf16": m.MB_PREC_BF16, "fp8": m.MB_PREC_FP8}[prec]
    a, b = teacher_params(), other_params(teacher_params(), 5)
    net, fresh = make_net(T, code, a), make_net(T, code, b)
    for n in (net, fresh):
        if prec == "fp8":
            calibrate(n, 9100)
    _, outs, blocks = batch_of(9000)
    old = run_batch(net, outs, blocks)
    net.load(b)
    if prec == "fp8":
        calibrate(net, 9100)
    got = run_batch(net, outs, blocks)
    for g, w, p, o in zip(got, run_batch(fresh, outs, blocks), run_batch(net, outs, blocks, True), old):
        assert np.abs(g - o).max() > 1e-3
        np.testing.assert_array_equal(g, w)
        np.testing.assert_array_equal(g, p)
    net.close()
    fresh.close()


def test_batch_after_a_second_calibration_uses_its_scales():
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    net = make_net(T, m.MB_PREC_FP8, teacher_params())
    calibrate(net, 9100)
    _, outs, blocks = batch_of(9000)
    run_batch(net, outs, blocks)
    calibrate(net, 9200, gain=2)
    got = run_batch(net, outs, blocks)
    for g, p in zip(got, run_batch(net, outs, blocks, True)):
        np.testing.assert_array_equal(g, p)
    net.close()


# --- calls captured in a caller's own graph -------------------------------------------------------

VOL = (2, 70, 140)


def net_and_other(layers, code, params, seed):
    """A net with its weights, a second one with others, and those."""
    from paper_1612_02120_gb300 import build
    build.build()
    b = other_params(params, seed)
    return make_net(layers, code, params), make_net(layers, code, b), b


def captured_volume(net, shape=VOL, sub=1):
    """A captured mb_infer_volume of `shape` on new bytes, its output, and the same call made at once."""
    import torch
    from paper_1612_02120_gb300 import membrane as m
    x = torch.from_numpy(synth.em_volume(9300, *shape)).cuda()
    z, h, w = shape
    out = torch.zeros((z, -(-h // sub), -(-w // sub)), device="cuda")

    def call(n, o):
        st = torch.cuda.current_stream()
        if sub == 1:
            m.mb_infer_volume(n.handle, x, z, h, w, o, stream=st)
        else:
            m.mb_infer_volume_subsampled(n.handle, x, z, h, w, sub, o, stream=st)

    call(net, out)  # the workspace grows outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(net, out)

    def replayed():
        out.fill_(-1.0)
        graph.replay()
        torch.cuda.synchronize()
        return out.cpu().numpy()

    def at_once(n):
        o = torch.full_like(out, -2.0)
        call(n, o)
        torch.cuda.synchronize()
        return o.cpu().numpy()

    return replayed, at_once


def check_replay(net, fresh, new, prepare=lambda n: None, **kw):
    for n in (net, fresh):
        prepare(n)
    replayed, at_once = captured_volume(net, **kw)
    old = replayed()
    np.testing.assert_array_equal(old, at_once(net))
    net.load(new)
    prepare(net)
    got = replayed()
    assert np.abs(got - old).max() > 1e-3
    np.testing.assert_array_equal(got, at_once(fresh))
    np.testing.assert_array_equal(at_once(net), got)
    net.close()
    fresh.close()


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
def test_captured_teacher_follows_a_reload(prec):
    from paper_1612_02120_gb300 import membrane as m
    code = {"bf16": m.MB_PREC_BF16, "fp8": m.MB_PREC_FP8}[prec]
    check_replay(*net_and_other(T, code, teacher_params(), 6),
                 prepare=(lambda n: calibrate(n, 9100)) if prec == "fp8" else (lambda n: None))


@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("sub", [1, 2])
def test_captured_fastmemb_follows_a_reload(prec, sub):
    from paper_1612_02120_gb300 import membrane as m
    code = {"bf16": m.MB_PREC_BF16, "fp16": m.MB_PREC_FP16}[prec]
    check_replay(*net_and_other(synth.FASTMEMB, code, synth.init_params(synth.FASTMEMB, 99, bias_std=0.01), 7), sub=sub)


@pytest.mark.parametrize("kind", ["teacher", "fastmemb", "student", "student_bf16"])
def test_captured_fp32_and_student_calls_follow_a_reload(kind):
    from paper_1612_02120_gb300 import membrane as m
    layers, code, params = {
        "teacher": (T, m.MB_PREC_FP32, teacher_params()),
        "fastmemb": (synth.FASTMEMB, m.MB_PREC_FP32, synth.init_params(synth.FASTMEMB, 99, bias_std=0.01)),
        "student": (synth.STUDENT, m.MB_PREC_FP32, student_params()),
        "student_bf16": (synth.STUDENT, m.MB_PREC_BF16, student_params())}[kind]
    check_replay(*net_and_other(layers, code, params, 8))


def test_captured_fp32_call_follows_weights_that_the_split_layers_refuse():
    """The new weights are the other net's with the first layer times 2^104 and the second over 2^104: the
    same network exactly, but beyond the bound of the split layers, so later calls take the CUDA cores. The
    captured call keeps its layers and gets the new weights; 2e-6 is the two paths' distance (see
    test_gpu_f32_tc)."""
    from paper_1612_02120_gb300 import membrane as m
    net, fresh, b = net_and_other(T, m.MB_PREC_FP32, teacher_params(), 8)
    replayed, at_once = captured_volume(net)
    old = replayed()
    big = b.copy()
    big[:832] *= np.float32(2.0 ** 104)
    big[832:832 + 25600] /= np.float32(2.0 ** 104)
    net.load(big)
    got = replayed()
    assert np.abs(got - old).max() > 1e-3
    assert np.abs(got - at_once(fresh)).max() <= 2e-6
    assert np.abs(at_once(net) - at_once(fresh)).max() <= 2e-6
    net.close()
    fresh.close()
