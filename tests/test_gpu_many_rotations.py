"""A call's memory does not grow with its rotations times the volume's sides, and a
call counted in several parts gives each rotation its own result."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_many_rotations():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_10156_gb300 import cs_ngf as cs
    dims, R = (6, 6, 250), 200_000
    gen = torch.Generator(device="cuda").manual_seed(3)
    A, B = (torch.rand(dims, generator=gen, device="cuda") for _ in range(2))
    M = torch.ones(dims, dtype=torch.uint8, device="cuda")
    half = np.random.default_rng(4).uniform(-0.3, 0.3, R)
    quats = np.stack([np.cos(half), np.sin(half), 0 * half, 0 * half], axis=1)     # about the long axis
    f = cs.prepare_fixed(A, M)
    sc = torch.empty(R, device="cuda")
    sh = torch.empty((R, 3), dtype=torch.int32, device="cuda")
    f.score_rotations(B, M, quats[:64], out_score=sc[:64], out_shift=sh[:64])
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    f.score_rotations(B, M, quats, out_score=sc, out_shift=sh)
    torch.cuda.synchronize()
    # 108 bytes a rotation, and 263 counts for 8192 of them: 30 MB; 210 MB with counts for all
    assert free - torch.cuda.mem_get_info()[0] < 100e6
    sc, sh = sc.cpu().numpy(), sh.cpu().numpy()
    assert np.isfinite(sc).all()
    for r0 in (0, 8184, 16380, 196_600, R - 8):
        s, c = [t.cpu().numpy() for t in f.score_rotations(B, M, quats[r0:r0 + 16])]
        np.testing.assert_allclose(sc[r0:r0 + 16], s, rtol=1e-5)
        np.testing.assert_array_equal(sh[r0:r0 + 16], c)
