"""Waits of the transform passes that run out: the pass ends by itself, the device
stays usable and the error reaches the caller."""
import ctypes

import pytest

from tests import native_util

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


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
