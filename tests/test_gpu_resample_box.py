"""cs_ngf_resample leaves nothing of its mask behind: the next call's mask counts
look at the next call's mask only."""
import ctypes

import numpy as np
import pytest

from paper_2110_10156_gb300 import synth
from tests import native_util

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_resample_leaves_no_mask_box(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_10156_gb300 import cs_ngf as cs
    flags = native_util.load("handle_flags.cu", tmp_path, ["-ldl"])
    p = synth.small_pair(29, (20, 18, 22), n_rot=2, masks="full")
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    f = cs.prepare_fixed(dev(p.A), dev(p.MA))
    box = (ctypes.c_int * 6)()
    for call in (lambda: f.score_rotations(dev(p.B), dev(p.MB), p.quats), lambda: f.resample(dev(p.B), dev(p.MB), p.quats[0])):
        call()
        assert flags.read_mask_box(f._h, box) == 0
        assert list(box) == [0] * 6
