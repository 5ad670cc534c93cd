"""A call's launches may begin while the one before still ends. Calls queued without a host
synchronisation between them share the net's workspace, so each launch has to wait for all that the
earlier ones read and write: queued calls give exactly what calls on their own give, also on two streams
(a net each) and replayed from a captured CUDA graph with new input bytes."""
import numpy as np
import pytest

import synth
from _common import infer, make_net, teacher_params

pytestmark = pytest.mark.gpu

CASES = {
    "fastmemb_bf16": (synth.FASTMEMB, "MB_PREC_BF16", (1, 90, 150)),
    "fastmemb_fp16_many_rows": (synth.FASTMEMB, "MB_PREC_FP16", (3, 400, 257)),
    "fastmemb_fp32": (synth.FASTMEMB, "MB_PREC_FP32", (2, 64, 140)),
    "teacher_fp32": (synth.TEACHER, "MB_PREC_FP32", (2, 50, 300)),
}


def net_of(name):
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    layers, prec, shape = CASES[name]
    params = teacher_params() if layers is synth.TEACHER else synth.init_params(layers, 99, bias_std=0.01)
    return make_net(layers, getattr(m, prec), params), shape


@pytest.mark.parametrize("name", list(CASES))
def test_queued_calls_equal_single_calls(name):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    nets = [net_of(name)[0] for _ in range(2)]
    shape = CASES[name][2]
    vols = [synth.em_volume(8000 + i, *shape) for i in range(3)]
    want = [infer(nets[0], v) for v in vols]
    xs = [torch.from_numpy(v).cuda() for v in vols]
    streams = [torch.cuda.Stream() for _ in nets]
    outs = [[torch.empty(shape, dtype=torch.float32, device="cuda") for _ in range(6)] for _ in nets]
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


@pytest.mark.parametrize("name", list(CASES))
def test_captured_call_replays(name):
    import torch
    from paper_1612_02120_gb300 import membrane as m
    net, shape = net_of(name)
    vols = [synth.em_volume(8100 + i, *shape) for i in range(3)]
    want = [infer(net, v) for v in vols]
    x = torch.from_numpy(vols[0]).cuda()
    out = torch.zeros(shape, dtype=torch.float32, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        m.mb_infer_volume(net.handle, x, *shape, out, stream=torch.cuda.current_stream())
    for i in (1, 2, 0):
        x.copy_(torch.from_numpy(vols[i]))
        graph.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy(), want[i])
    net.close()
