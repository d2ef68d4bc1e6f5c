"""cp.async copies and their waits in the CUDA sources: cp.async.wait_group waits for
committed groups only, so a source that commits none has to use cp.async.wait_all."""
import os
import re

from paper_2110_10156_gb300 import build


def test_uncommitted_copies_are_waited_for_by_wait_all():
    text = {}
    for name in sorted(os.listdir(build.CSRC)):
        with open(os.path.join(build.CSRC, name)) as fh:
            text[name] = re.sub(r"//[^\n]*", "", fh.read())
    helpers = text["fft_core.cuh"]
    wait = re.search(r"void cp_async_wait_all\(\) \{([^}]*)\}", helpers).group(1)
    users = [n for n, t in text.items() if n != "fft_core.cuh" and re.search(r"cp_async\d+\(", t)]
    for n in users:
        assert "cp_async_wait_all()" in text[n], n
        if "cp_async_commit()" not in text[n]:
            assert "cp.async.wait_all" in wait, n
