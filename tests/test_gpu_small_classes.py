"""Rotations of a small volume that need different lengths: a class of their own
costs more in launches than its shorter transforms save, so they share one."""
import numpy as np
import pytest

from paper_2110_10156_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_10156_gb300 import build
    build.build()
    from paper_2110_10156_gb300 import cs_ngf
    return cs_ngf


def test_small_volume_takes_one_class(cs):
    dims = (24, 24, 24)
    p = synth.small_pair(57, dims, masks="full", n_rot=2)
    M = np.zeros(dims, np.uint8)
    M[6:18, 8:16, 8:16] = 1
    half = np.sqrt(0.5)
    a, b = [1.0, 0.0, 0.0, 0.0], [half, half, 0.0, 0.0]       # identity, a quarter turn that swaps z and y
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    f = cs.prepare_fixed(dev(p.A), dev(M))
    alone, pads = [], set()
    for q in (a, b):
        sc, sh = f.score_rotations(dev(p.B), dev(M), [q])
        alone.append((float(sc[0]), sh[0].tolist()))
        pads.add(f.transform_classes()[0][0])
    assert len(pads) == 2                                       # they need different lengths
    sc, sh = [t.cpu().numpy() for t in f.score_rotations(dev(p.B), dev(M), [a, b] * 13)]
    (pad, n), = f.transform_classes()
    assert n == 26 and all(pad[k] == max(q[k] for q in pads) for k in range(3))
    for r in range(26):
        assert abs(sc[r] - alone[r % 2][0]) <= 1e-5 * abs(alone[r % 2][0])
        assert sh[r].tolist() == alone[r % 2][1]
