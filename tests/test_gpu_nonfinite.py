"""NaN and infinities: no influence where no gradient under a mask reads them, no
valid shift where one does (the convention include/cs_ngf.h states)."""
import numpy as np
import pytest

from paper_2110_10156_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FORMS = [dict(), dict(pad_mode="full"), dict(precision="bf16"), dict(precision="fp16", tensor_cores=False),
         dict(measure="unsquared"), dict(autotune="alternative")]


@pytest.fixture(scope="module")
def cs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_10156_gb300 import build
    build.build()
    from paper_2110_10156_gb300 import cs_ngf
    return cs_ngf


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def pair():
    dims = (26, 25, 27)
    p = synth.small_pair(61, dims, masks="full", n_rot=18)       # more than 16: cells far from the mask are left out
    M = np.zeros(dims, np.uint8)
    M[9:18, 8:17, 9:17] = 1
    far = np.ones(dims, bool)
    far[5:22, 4:21, 5:21] = False                 # four voxels and more from the mask: a sample reaches two cells
    return p, M, far


@pytest.mark.parametrize("kw", FORMS)
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_no_influence_outside_the_masks(cs, kw, value):
    p, M, far = pair()
    A, B = p.A.copy(), p.B.copy()
    A[far] = value
    B[far] = -value
    for quats in (p.quats, p.quats[:3]):
        ref = cs.prepare_fixed(dev(p.A), dev(M), **kw)
        want = [t.cpu().numpy() for t in ref.score_rotations(dev(p.B), dev(M), quats)]
        f = cs.prepare_fixed(dev(A), dev(M), **kw)
        got = [t.cpu().numpy() for t in f.score_rotations(dev(B), dev(M), quats)]
        assert np.isfinite(want[0]).any()
        np.testing.assert_array_equal(got[0], want[0])
        np.testing.assert_array_equal(got[1], want[1])


@pytest.mark.parametrize("kw", FORMS)
@pytest.mark.parametrize("side", ["A", "B"])
def test_no_valid_shift_where_a_gradient_reads_it(cs, kw, side):
    p, M, _ = pair()
    v = dict(A=p.A.copy(), B=p.B.copy())
    v[side][13, 12, 12] = np.nan
    f = cs.prepare_fixed(dev(v["A"]), dev(M), **kw)
    sc, sh = [t.cpu().numpy() for t in f.score_rotations(dev(v["B"]), dev(M), p.quats)]
    assert np.isneginf(sc).all() and (sh == 0).all()
    assert f.align(dev(v["B"]), dev(M), p.quats) == (-np.inf, -1, (0, 0, 0))
