"""A caller may write the fixed volume's arrays again, on any stream, once
cs_ngf_prepare_fixed or cs_ngf_update_fixed has returned."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("pad_mode", ["bound", "full"])
@pytest.mark.parametrize("call", ["prepare_fixed", "update_fixed"])
def test_fixed_volume_overwritten_on_another_stream(cs, pad_mode, call):
    dims = (160, 176, 168)
    gen = torch.Generator(device="cuda").manual_seed(5)
    rand = lambda: torch.rand(dims, generator=gen, device="cuda")
    first, A, junk, B = rand(), rand(), rand(), rand()
    M = torch.ones(dims, dtype=torch.uint8, device="cuda")
    q = [[1.0, 0.0, 0.0, 0.0]]
    ref = cs.prepare_fixed(A, M, pad_mode=pad_mode)
    want = [t.cpu().numpy() for t in ref.score_rotations(B, M, q)]
    ref.release()
    other, busy = torch.cuda.Stream(priority=-1), torch.cuda.Stream()
    X = torch.rand(8192, 8192, device="cuda").bfloat16()
    with torch.cuda.stream(busy):
        X @ X
    if call == "update_fixed":
        f = cs.prepare_fixed(first, M, pad_mode=pad_mode)
        f.score_rotations(B, M, q)               # the lengths the next call keeps
    A2, M2 = A.clone(), M.clone()
    with torch.cuda.stream(other):               # its kernels are loaded
        A2.copy_(A)
        M2.copy_(M)
        M.clone().zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(busy):                # about 50 ms: what the call leaves running takes its time
        for _ in range(80):
            X @ X
    if call == "update_fixed":
        f.update_fixed(A2, M2)
    else:
        f = cs.prepare_fixed(A2, M2, pad_mode=pad_mode)
    with torch.cuda.stream(other):
        A2.copy_(junk)
        M2.zero_()
    got = [t.cpu().numpy() for t in f.score_rotations(B, M, q)]
    torch.cuda.synchronize()
    f.release()
    np.testing.assert_array_equal(got[0], want[0])
    np.testing.assert_array_equal(got[1], want[1])
