"""The autotuner's cache: an entry that does not name the slices it was timed on (those of earlier versions,
timed on white noise, whose choice is slower on EM slices) is not taken over; the shape is timed again and its
entry added, and the old line stays in the file."""
import pytest

import synth
from _common import make_net, teacher_params

pytestmark = pytest.mark.gpu


def test_entry_without_a_workload_is_timed_again(tmp_path):
    import torch
    from paper_1612_02120_gb300 import build, membrane as m
    build.build()
    net, cache = make_net(synth.TEACHER, m.MB_PREC_BF16, teacher_params()), tmp_path / "tune.json"
    old = '{"key": "%s|bf16|2x300x260", "rows_per_item": 1024, "stages": 6, "ms": 0.1000}\n' % torch.cuda.get_device_name(0)
    cache.write_text(old)
    first = m.mb_autotune(net.handle, 2, 300, 260, str(cache))
    assert not first["from_cache"]
    again = m.mb_autotune(net.handle, 2, 300, 260, str(cache))
    assert again["from_cache"] and {**again, "from_cache": False} == first
    lines = cache.read_text().splitlines(keepends=True)
    assert lines[0] == old and len(lines) == 2
    net.close()
