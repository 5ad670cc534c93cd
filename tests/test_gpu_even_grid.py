"""The even split's launch size: the same maps, bitwise, whether a launch runs one CTA per SM cut anywhere,
the same number of CTAs per column, or round-robin items."""
import numpy as np
import pytest

import synth
from _common import infer, make_net, teacher_params

pytestmark = pytest.mark.gpu


# one row per CTA; a column split 152 ways; rows that do not divide; more columns than SMs
@pytest.mark.parametrize("shape", [(1, 8, 8), (1, 9, 119), (1, 153, 117), (1, 257, 237), (2, 31, 700), (40, 16, 500)])
def test_default_split_equals_round_robin_items(shape):
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    net = make_net(synth.TEACHER, m.MB_PREC_BF16, teacher_params())
    v = synth.em_volume(7600 + shape[1], *shape)
    got = infer(net, v)
    m.mb_set_tuning(net.handle, 64, 6)
    assert np.array_equal(got, infer(net, v))
    net.close()
