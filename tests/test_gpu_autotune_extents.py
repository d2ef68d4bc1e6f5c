"""The autotuner's table tells a pass on a half-filled input from one on a fuller
one by what the pass transforms: masks' extents, not the volume's sides."""
import numpy as np
import pytest

from paper_2110_10156_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_table_follows_the_extents():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_10156_gb300 import cs_ngf as cs
    cs.tuning_reset()
    n = 40
    p = synth.small_pair(33, (n, n, n), masks="full", n_rot=2)
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    q = [[1.0, 0.0, 0.0, 0.0]]

    def cube(m):                                  # slabs 0 .. m - 1 of each axis
        M = np.zeros((n, n, n), np.uint8)
        M[:m, :m, :m] = 1
        return dev(M)

    A, B = dev(p.A), dev(p.B)
    f = cs.prepare_fixed(A, cube(16), autotune=True)
    f.align(B, cube(16), q)
    assert f.transform_classes() == [((64, 64, 64), 1)]
    half = lambda: {(e["stage"], e["half_input"]) for e in cs.tuning() if e["stage"] in ("fwd_x", "fwd_y", "zmac")}
    assert half() == {("fwd_x", True), ("fwd_y", True), ("zmac", True)}     # 16 of 64, though the side is 40
    f.update_fixed(A, cube(38))
    got = f.align(B, cube(38), q)
    assert f.transform_classes() == [((64, 64, 64), 1)]                     # the same lengths, other extents
    assert half() == {(s, h) for s in ("fwd_x", "fwd_y", "zmac") for h in (True, False)}
    ref = cs.prepare_fixed(A, cube(38))
    want = ref.align(B, cube(38), q)
    assert got[1:] == want[1:] and abs(got[0] - want[0]) <= 1e-4 * abs(want[0])
    cs.tuning_reset()
