"""A fixed volume whose spectra could not be launched is not scored with the spectra
of the one before it."""
import os
import subprocess
import sys

import pytest

from paper_2110_10156_gb300 import build
from tests import native_util

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes, os
import numpy as np, torch
from paper_2110_10156_gb300 import cs_ngf as cs, synth
fail = ctypes.CDLL(os.environ["LD_PRELOAD"])
p, o = (synth.small_pair(s, (30, 29, 28), masks="full", n_rot=2) for s in (5, 6))   # 64-point lengths
dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
kw = dict(pad_mode=%r, autotune="alternative")
B, M = dev(p.B), dev(p.MB)
want = cs.prepare_fixed(dev(p.A), M, **kw).align(B, M, p.quats)
f = cs.prepare_fixed(dev(o.A), M, **kw)
f.align(B, M, p.quats)
A = dev(p.A)

def status(call):
    try:
        return call()
    except cs.CsNgfError as e:
        return e.status

fail.arm_failure()
assert status(lambda: f.update_fixed(A, M)) == cs.ECUDA
got = status(lambda: f.align(B, M, p.quats))
if kw["pad_mode"] == "full":                     # no copies to compute them from
    assert got == cs.ECUDA, got
    f.update_fixed(A, M)
    got = f.align(B, M, p.quats)
assert got == want, (got, want)
print("sound")
"""


@pytest.mark.parametrize("pad_mode", ["bound", "full"])
def test_spectra_that_were_not_launched(pad_mode, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = native_util.compile_shared("fail_spectra.cu", tmp_path, ["-ldl"])
    env = dict(os.environ, LD_PRELOAD=lib, CS_NGF_LIB=build.LIB)
    out = subprocess.run([sys.executable, "-c", CHILD % pad_mode], cwd=ROOT, env=env, capture_output=True, text=True,
                         timeout=120)
    assert out.returncode == 0 and "sound" in out.stdout, out.stderr
