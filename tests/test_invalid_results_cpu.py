"""NaN scores are the library's mark of invalid results (include/cs_ngf.h): a long
job neither saves nor returns them, and a rank does not merge past them."""
import numpy as np
import pytest

from paper_2110_10156_gb300 import resume, shard
from paper_2110_10156_gb300.synth import random_quaternions


class Scorer:
    dims = (16, 16, 16)

    def __init__(self, bad_call=None):
        self.calls, self.bad_call = 0, bad_call

    def score_rotations(self, B, MB, q):
        self.calls += 1
        s = np.linspace(0.1, 0.2, len(q)).astype(np.float32)
        if self.calls == self.bad_call:
            s[:] = np.nan
        return s, np.zeros((len(q), 3), np.int32)


def test_resumable_job_scores_an_invalid_chunk_again(tmp_path):
    q = random_quaternions(np.random.default_rng(2), 12)
    path = str(tmp_path / "ck.npz")
    with pytest.raises(RuntimeError, match="invalid"):
        resume.score_rotations_resumable(Scorer(bad_call=2), None, None, q, path, chunk=4)
    rest = Scorer()
    s, _ = resume.score_rotations_resumable(rest, None, None, q, path, chunk=4)
    assert rest.calls == 2 and not np.isnan(s).any()


def test_a_rank_does_not_merge_invalid_scores():
    ok = np.array([0.1, -np.inf, 0.3])
    assert shard.local_best(ok, np.zeros((3, 3), int), 5) == (0.3, 7, (0, 0, 0))
    with pytest.raises(RuntimeError, match="invalid"):
        shard.local_best(np.array([0.1, np.nan, 0.3]), np.zeros((3, 3), int), 5)
