"""The hash that ties a DRAM traffic summary to the kernels covers every source a
scoring kernel is built from."""
import importlib.util
import os
import re
import shutil
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_hash_covers_the_included_sources(monkeypatch, tmp_path):
    spec = importlib.util.spec_from_file_location("bench_sources", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    monkeypatch.setitem(sys.modules, "bench_sources", bench)
    spec.loader.exec_module(bench)
    csrc = tmp_path / "paper_2110_10156_gb300" / "csrc"
    shutil.copytree(os.path.join(ROOT, "paper_2110_10156_gb300", "csrc"), csrc)
    # what the pass sources include, directly or through another header
    seen, todo = set(), ["passes_16.cu", "elem.cu", "cs_ngf.cu"]
    while todo:
        name = todo.pop()
        if name in seen or not (csrc / name).exists():
            continue
        seen.add(name)
        todo += re.findall(r'#include "([^"]+)"', (csrc / name).read_text())
    assert "zpass.cuh" in seen and len(seen) > 6
    for name in sorted(seen):
        monkeypatch.setattr(bench, "ROOT", str(tmp_path))
        bench._SOURCE_HASH.clear()
        before = bench.kernel_source_hash()
        with open(csrc / name, "a") as fh:
            fh.write("// changed\n")
        bench._SOURCE_HASH.clear()
        assert bench.kernel_source_hash() != before, name
