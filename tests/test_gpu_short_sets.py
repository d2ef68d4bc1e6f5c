"""Rotation counts around the z pass's sets of four: each rotation's result is what
it is among other counts, whatever slots of the last set are empty."""
import numpy as np
import pytest

from paper_2110_10156_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kw", [dict(), dict(pad_mode="full"), dict(precision="bf16"), dict(precision="fp16", tensor_cores=False),
                                dict(measure="unsquared", pad_mode="full")])
def test_results_do_not_depend_on_the_empty_slots(kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_10156_gb300 import cs_ngf as cs
    p = synth.small_pair(77, (40, 37, 42), masks="full", n_rot=12)
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    f = cs.prepare_fixed(dev(p.A), dev(p.MA), **kw)
    B, MB = dev(p.B), dev(p.MB)
    # one rotation twelve times over: one class, the same lengths for every count
    q = np.repeat(p.quats[:1], 12, axis=0)
    want = [t.cpu().numpy() for t in f.score_rotations(B, MB, q)]
    for n in range(2, 12):                       # even and odd, with every number of empty slots
        got = [t.cpu().numpy() for t in f.score_rotations(B, MB, q[:n])]
        k = n // 2 * 2                           # an odd last mask is transformed alone: its last bits may differ
        np.testing.assert_array_equal(got[0][:k], want[0][:k])
        np.testing.assert_array_equal(got[1], want[1][:n])
        np.testing.assert_allclose(got[0][k:], want[0][k:n], rtol=1e-5)
