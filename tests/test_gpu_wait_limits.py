"""Waits of the transform passes that run out: the pass ends by itself, the device
stays usable and the error reaches the caller."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2110_10156_gb300 import build, synth
from tests import native_util

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CALLS = ["search", "server"]


@pytest.fixture(scope="module")
def passes(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return native_util.load("wait_limits.cu", tmp_path_factory.mktemp("native"))


# a pass's copies, in the order the blocks issue them: 0 is a first one, the others
# lie in later groups (y: 64 copies a group and block row) and fields (z)
@pytest.mark.parametrize("p,drop", [(0, 0), (0, 150), (0, 400), (0, 610), (1, 0), (1, 200), (1, 700), (1, 1500)])
def test_a_missing_copy_ends_the_pass_with_its_flag_set(passes, p, drop):
    flag = ctypes.c_int(-1)
    assert passes.run_pass(p, -1, ctypes.byref(flag)) == 0 and flag.value == 0
    assert passes.run_pass(p, drop, ctypes.byref(flag)) == 0 and flag.value == 1
    assert passes.run_pass(p, -1, ctypes.byref(flag)) == 0 and flag.value == 0


@pytest.fixture(scope="module")
def flags(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return native_util.load("handle_flags.cu", tmp_path_factory.mktemp("native"))


@pytest.mark.parametrize("pad_mode", ["bound", "full"])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_invalid_spectra_reach_every_call(flags, pad_mode, precision):
    from paper_2110_10156_gb300 import cs_ngf as cs
    p = synth.small_pair(19, (12, 14, 13), n_rot=5)
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    A, MA, B, MB = dev(p.A), dev(p.MA), dev(p.B), dev(p.MB)
    f = cs.prepare_fixed(A, MA, pad_mode=pad_mode, precision=precision)
    want = f.align(B, MB, p.quats)

    def raised():
        if pad_mode == "bound":                  # the call after one that failed computes the spectra again
            assert f.align(B, MB, p.quats) == want
        assert flags.raise_spectra_flag(f._h) == 0

    raised()
    sc, sh = f.score_rotations(B, MB, p.quats)
    assert torch.isnan(sc).all() and (sh == 0).all()
    raised()
    assert torch.isnan(f.score_map(B, MB, p.quats[0])).all()
    for call in (lambda: f.align(B, MB, p.quats), lambda: f.score_rotations_host(p.B, p.MB, p.quats)):
        raised()
        with pytest.raises(cs.CsNgfError) as e:
            call()
        assert e.value.status == cs.ECUDA and "timed out" in str(e.value)
    if pad_mode == "full":                       # nothing to compute them from again
        with pytest.raises(cs.CsNgfError):
            f.align(B, MB, p.quats)
        f.update_fixed(A, MA)
    assert f.align(B, MB, p.quats) == want       # not blamed for the calls before it


def test_a_flag_of_an_asynchronous_call_is_not_the_next_ones(flags):
    from paper_2110_10156_gb300 import cs_ngf as cs
    p = synth.small_pair(19, (12, 14, 13), n_rot=5)
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    f = cs.prepare_fixed(dev(p.A), dev(p.MA))
    want = f.align(dev(p.B), dev(p.MB), p.quats)
    assert flags.raise_spectra_flag(f._h) == 0
    sc, _ = f.score_rotations(dev(p.B), dev(p.MB), p.quats)
    torch.cuda.synchronize()
    assert torch.isnan(sc).all()
    assert f.align(dev(p.B), dev(p.MB), p.quats) == want


@pytest.fixture(scope="module")
def noalloc(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return native_util.load("wait_limits_noalloc.cu", tmp_path_factory.mktemp("native"),
                            [os.path.join(build.CSRC, "elem.cu")])


def test_allocation_free_results_say_that_a_wait_ran_out(noalloc):
    p = synth.small_pair(23, (8, 7, 6), n_rot=3, masks="full")
    dev = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p.A, p.MA, p.B, p.MB)]
    quats = np.ascontiguousarray(p.quats, dtype=np.float64)
    R = len(quats)
    copies = ctypes.c_int(0)

    def run(drop):
        assert noalloc.set_drop(drop, ctypes.byref(copies)) == 0
        sc = torch.zeros(R, device="cuda")
        sh = torch.full((R, 3), 9, dtype=torch.int32, device="cuda")
        st = noalloc.cs_ngf_score_rotations_noalloc(
            *(ctypes.c_void_p(t.data_ptr()) for t in dev), (ctypes.c_int32 * 3)(8, 7, 6), ctypes.c_float(1e-5),
            ctypes.c_float(0.5), quats.ctypes.data_as(ctypes.c_void_p), R, ctypes.c_void_p(sc.data_ptr()),
            ctypes.c_void_p(sh.data_ptr()), None)
        assert st == 0
        torch.cuda.synchronize()
        assert noalloc.set_drop(-1, ctypes.byref(copies)) == 0
        return sc.cpu().numpy(), sh.cpu().numpy(), copies.value

    want, shift, total = run(-1)
    assert np.isfinite(want).all() and total > 0
    sc, sh, _ = run(0)                           # a copy of the fixed spectra: every rotation
    assert np.isnan(sc).all() and (sh == 0).all()
    sc, sh, _ = run(total - 1)                   # the last rotation's last copy
    np.testing.assert_array_equal(sc[:-1], want[:-1])
    np.testing.assert_array_equal(sh[:-1], shift[:-1])
    assert np.isnan(sc[-1]) and (sh[-1] == 0).all()
    again, _, _ = run(-1)
    np.testing.assert_array_equal(again, want)


CHILD = """
import numpy as np, torch
from paper_2110_10156_gb300 import cs_ngf as cs, synth
p = synth.small_pair(19, (12, 14, 13), n_rot=5)
dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
if %r == "search":
    try:
        cs.global_align(dev(p.A), dev(p.MA), dev(p.B), dev(p.MB), schedule=[(1.0, 1, 20.0, 5, 1)], seed=1)
        print("status", 0)
    except cs.CsNgfError as e:
        print("status", e.status, e)
else:
    srv = cs.Server()
    print("status", srv.wait(srv.submit(p.A, p.MA, p.B, p.MB, p.quats))["status"])
    srv.close()
"""


@pytest.mark.parametrize("call", CALLS)
def test_handles_made_inside_the_library(call, tmp_path):
    """The search and the server prepare handles of their own: a child process whose
    library finds their flag raised."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_10156_gb300 import cs_ngf as cs
    lib = native_util.compile_shared("handle_flags.cu", tmp_path, ["-ldl"])
    env = dict(os.environ, LD_PRELOAD=lib, CS_NGF_LIB=build.LIB)
    out = subprocess.run([sys.executable, "-c", CHILD % call], cwd=ROOT, env=env, capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stderr
    assert f"status {cs.ECUDA}" in out.stdout, out.stdout
