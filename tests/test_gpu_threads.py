"""Handles of two host threads whose passes take different amounts of shared memory at
the same FFT lengths."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_two_threads_two_extents(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_10156_gb300 import cs_ngf as cs
    q = np.array([[1.0, 0.0, 0.0, 0.0], [0.0, 1.0, 0.0, 0.0]])
    errors, handles = [], []
    for n in (85, 96) * 3:                        # 2n - 1 <= 192 for both: one length, two extents
        dims = (n, 12, 6)
        gen = torch.Generator(device="cuda").manual_seed(n)
        A, B = (torch.rand(dims, generator=gen, device="cuda") for _ in range(2))
        M = torch.ones(dims, dtype=torch.uint8, device="cuda")
        f = cs.prepare_fixed(A, M, pad_mode="full", precision=precision, batch=2)
        handles.append((f, B, M, torch.cuda.Stream(), [t.clone() for t in f.score_rotations(B, M, q)]))
    assert handles[0][0].max_pad == handles[1][0].max_pad

    def work(f, B, M, stream, want):
        try:
            sc, sh = torch.empty_like(want[0]), torch.empty_like(want[1])
            for _ in range(3000):                 # enqueued without a wait for the results: launch after launch
                f.score_rotations(B, M, q, out_score=sc, out_shift=sh, stream=stream)
            stream.synchronize()
            if not (torch.equal(sc, want[0]) and torch.equal(sh, want[1])):
                errors.append((sc, sh, want))
        except Exception as e:
            errors.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=h) for h in handles]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
