"""Transforms of the masks' boxes (bound-limited padding, FP32): the lengths the
boxes allow, and scores and maps against the oracle's full-length maps, for
boxes in a corner, thinner than a tile, of one voxel, touching the faces, and
filling the volume; and the same calls in the forms that keep the rule's
lengths (16-bit storage, autotuning)."""
import numpy as np
import pytest

from oracle import cs_ngf_oracle as O
from paper_2110_10156_gb300 import synth
from tests.parity_util import TAU_FP32, check_best_against_map, check_maps

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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def box_mask(dims, lo, hi):
    m = np.zeros(dims, np.uint8)
    m[tuple(slice(a, b + 1) for a, b in zip(lo, hi))] = 1
    return m


def slabs(M, ax):
    return M.astype(np.int64).sum(axis=tuple(i for i in range(3) if i != ax))


def need(MA, Mh, gamma=0.5):
    """Per axis the points that keep the admitted shifts alias-free between the
    two masks' boxes; None if an axis admits none."""
    thr = O.overlap_threshold(int(MA.sum()), int(Mh.sum()), gamma)
    out = []
    for ax in range(3):
        a, b = slabs(MA, ax), slabs(Mh, ax)
        n = len(a)
        ok = [c for c in range(-(n - 1), n)
              if np.minimum(a[max(0, -c):min(n, n - c)], b[max(0, c):min(n, n + c)]).sum() >= thr]
        if not ok:
            return None
        a, b = np.nonzero(a)[0], np.nonzero(b)[0]
        out.append(max(b[-1] - a[0] - min(ok), max(ok) - b[0] + a[-1], b[-1] - b[0], a[-1] - a[0]) + 1)
    return out


# dims, box of M_A, box of M_B
CASES = [
    ((24, 22, 26), ((0, 0, 0), (8, 7, 9)), ((12, 10, 14), (23, 21, 25))),          # opposite corners
    ((33, 40, 30), ((10, 12, 9), (20, 14, 9)), ((8, 15, 5), (19, 18, 22))),        # thin boxes
    ((18, 17, 20), ((9, 8, 9), (9, 8, 9)), ((4, 4, 4), (13, 12, 15))),             # one voxel
    ((50, 45, 48), ((5, 0, 11), (44, 44, 36)), ((0, 7, 0), (49, 30, 47))),         # to the faces
    ((20, 33, 27), ((0, 0, 0), (19, 32, 26)), ((0, 0, 0), (19, 32, 26))),          # the whole volume
    ((70, 12, 9), ((30, 2, 1), (66, 9, 8)), ((2, 3, 0), (40, 11, 7))),             # one long axis
]


@pytest.mark.parametrize("measure", ["squared", "unsquared"])
@pytest.mark.parametrize("dims,box_a,box_b", CASES)
def test_boxes_match_oracle(cs, dims, box_a, box_b, measure):
    p = synth.small_pair(70 + sum(dims), dims, masks="full", n_rot=5)
    MA, MB = box_mask(dims, *box_a), box_mask(dims, *box_b)
    half = np.sqrt(0.5)
    quats = np.concatenate([p.quats, [[half, 0.0, 0.0, half], [0.0, 1.0, 0.0, 0.0]]])
    f = cs.prepare_fixed(dev(p.A), dev(MA), measure=measure, batch=4)
    sc, sh = [t.cpu().numpy() for t in f.score_rotations(dev(p.B), dev(MB), quats)]
    ran = [c for c, k in f.transform_classes() for _ in range(k)]
    assert len(ran) == len(quats)
    needs, low = [], [None] * 3
    for r, q in enumerate(quats):
        _, Mh = O.resample(p.B, MB, q)
        needs.append(need(MA, Mh))
        omap, _ = O.score_map(p.A, MA, p.B, MB, q, measure=measure)
        assert np.isfinite(sc[r]) == np.isfinite(omap).any()
        if np.isfinite(sc[r]):
            check_best_against_map(omap, sc[r], sh[r])
        gmap = f.score_map(dev(p.B), dev(MB), q).cpu().numpy()
        np.testing.assert_array_equal(np.isfinite(gmap), np.isfinite(omap))
        if np.isfinite(omap).any():
            check_maps(omap, gmap)
            (one, k), = f.transform_classes()
            assert k == 1 and all(v >= n for v, n in zip(one, needs[-1]))
    known = [n for n in needs if n is not None]
    for a in range(3):
        assert max(c[a] for c in ran) >= max(n[a] for n in known)
        assert all(c[a] <= m for c, m in zip(ran, [f.max_pad[a]] * len(ran)))


@pytest.mark.parametrize("kw", [dict(precision="bf16"), dict(precision="fp16", tensor_cores=False),
                                dict(autotune="alternative"), dict(autotune=True)])
def test_forms_that_keep_the_rules_lengths(cs, kw):
    dims, (a, b) = (33, 40, 30), (((10, 12, 9), (20, 24, 19)), ((8, 15, 5), (19, 28, 22)))
    p = synth.small_pair(83, dims, masks="full", n_rot=5)
    MA, MB = box_mask(dims, *a), box_mask(dims, *b)
    f = cs.prepare_fixed(dev(p.A), dev(MA), batch=4, **kw)
    sc, sh = [t.cpu().numpy() for t in f.score_rotations(dev(p.B), dev(MB), p.quats)]
    assert sorted(f.transform_classes()) == sorted(f.length_classes())
    for r, q in enumerate(p.quats):
        omap, _ = O.score_map(p.A, MA, p.B, MB, q)
        check_best_against_map(omap, sc[r], sh[r], tau=TAU_FP32 if "precision" not in kw else 1e-2)


def test_another_fixed_volume_with_a_larger_box(cs):
    """update_fixed to a mask whose box no longer fits the lengths in use."""
    p = synth.small_pair(91, (40, 40, 40), masks="full", n_rot=3)
    small = box_mask((40, 40, 40), (15, 16, 17), (20, 22, 21))
    f = cs.prepare_fixed(dev(p.A), dev(small))
    f.score_rotations(dev(p.B), dev(small), p.quats)
    assert max(f.transform_classes()[-1][0]) < 40
    f.update_fixed(dev(p.A), dev(p.MA))
    sc, sh = [t.cpu().numpy() for t in f.score_rotations(dev(p.B), dev(p.MB), p.quats)]
    g = cs.prepare_fixed(dev(p.A), dev(p.MA))
    s2, c2 = [t.cpu().numpy() for t in g.score_rotations(dev(p.B), dev(p.MB), p.quats)]
    np.testing.assert_array_equal(sc, s2)
    np.testing.assert_array_equal(sh, c2)


# lengths only box transforms take (csrc/fft_core.cuh box_only), and their neighbours below
BOX_LENGTHS = {24: 16, 48: 40, 56: 48, 72: 64, 96: 80, 112: 100, 120: 112, 144: 128, 168: 160, 180: 168,
               240: 216, 280: 256, 300: 280}


@pytest.mark.parametrize("P", sorted(BOX_LENGTHS))
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_box_only_lengths_match_oracle(cs, P, axis):
    """Full masks admit shifts to half the side, so a side of 2P/3 needs P points;
    the map and the best shift of both rotations against the oracle."""
    dims = [7, 9, 6]
    dims[axis] = max(n for n in range(2, P) if n + n // 2 <= P)
    p = synth.small_pair(300 + P + axis, tuple(dims), masks="full", n_rot=2)
    f = cs.prepare_fixed(dev(p.A), dev(p.MA))
    gmap = f.score_map(dev(p.B), dev(p.MB), [1.0, 0.0, 0.0, 0.0]).cpu().numpy()
    (ran, _), = f.transform_classes()
    assert ran[axis] == P
    check_maps(O.score_map(p.A, p.MA, p.B, p.MB, [1.0, 0.0, 0.0, 0.0])[0], gmap)
    sc, sh = [t.cpu().numpy() for t in f.score_rotations(dev(p.B), dev(p.MB), p.quats)]
    for r, q in enumerate(p.quats):
        check_best_against_map(O.score_map(p.A, p.MA, p.B, p.MB, q)[0], sc[r], sh[r])


@pytest.mark.parametrize("dims,R,kw", [((20, 23, 18), 131, {}), ((20, 23, 18), 65, dict(precision="bf16")),
                                       ((33, 30, 36), 290, dict(measure="unsquared"))])
def test_automatic_launch_groups_match_small_ones(cs, dims, R, kw):
    """Automatic handles score more than 32 rotations per launch group at short
    lengths: bit for bit what groups of eight give, for a class's odd rest too."""
    p = synth.small_pair(410 + R, dims, masks="full", n_rot=R)
    MA, MB = box_mask(dims, (4, 5, 3), (14, 17, 15)), box_mask(dims, (2, 6, 4), (15, 19, 14))
    a = cs.prepare_fixed(dev(p.A), dev(MA), **kw)
    b = cs.prepare_fixed(dev(p.A), dev(MA), batch=8, **kw)
    assert a.batch == 32
    for x, y in zip(a.score_rotations(dev(p.B), dev(MB), p.quats), b.score_rotations(dev(p.B), dev(MB), p.quats)):
        np.testing.assert_array_equal(x.cpu().numpy(), y.cpu().numpy())
