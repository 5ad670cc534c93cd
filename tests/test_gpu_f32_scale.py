"""FP32 nets whose layers live near the small end of FP32's range. A net whose first layer is scaled by
2^-118 and whose second layer by 2^118 is the same network exactly (powers of two commute with ReLU, max-out
and max-filters), and FP32 arithmetic keeps its accuracy there: the layers' sums lie at 2^-118, 31 binary
orders above FP32's smallest step. A split of the values in BF16 parts does not (BF16 ends at 2^-133).

Tolerance: no worse than the CUDA cores' FP32 FMAs by more than one rounding of a probability (6e-8); they run
the same network with the factors 2^104 and 2^-104 (beyond the range that the split layers take)."""
import numpy as np
import pytest

import oracle
import synth
from _common import infer, make_net, teacher_params

pytestmark = pytest.mark.gpu

NETS = {
    "teacher": (synth.TEACHER, teacher_params, 832, 25600),
    "fastmemb": (synth.FASTMEMB, lambda: synth.init_params(synth.FASTMEMB, synth.FASTMEMB_WEIGHT_SEED), 64 * 16 + 64,
                 64 * 32 * 16),
}


@pytest.mark.parametrize("name", list(NETS))
def test_small_layers_keep_fp32_accuracy(name):
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    layers, params, n1, n2 = NETS[name]
    params = params()
    def times(e):
        p = params.copy()
        p[:n1] *= np.float32(2.0 ** e)
        p[n1:n1 + n2] *= np.float32(2.0 ** -e)
        assert np.isfinite(p).all()
        return make_net(layers, m.MB_PREC_FP32, p)

    v = synth.em_volume(7600, 1, 40, 133)
    exact = oracle.forward_region(layers, params, v[0])
    fma, small = times(104), times(-118)
    ref, got = infer(fma, v)[0], infer(small, v)[0]
    assert np.abs(got - exact).max() <= np.abs(ref - exact).max() + 6e-8
    fma.close()
    small.close()
