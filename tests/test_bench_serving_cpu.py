"""The serving measurement's offered load: from warm jobs, whatever the first job of
each shape costs."""
import argparse
import importlib.util
import os
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


class FakeServer:
    """Each shape's first job takes 0.3 s, every later one next to nothing."""

    def __init__(self, **kw):
        self.seen, self.jobs = set(), []

    def submit(self, A, MA, B, MB, quats, **kw):
        self.jobs.append((A.shape, len(quats)))
        return len(self.jobs) - 1

    def wait(self, job, **kw):
        shape, _ = self.jobs[job]
        if shape not in self.seen:
            self.seen.add(shape)
            time.sleep(0.3)
        return dict(status=0, latency_ms=1.0)

    def close(self):
        pass


def test_capacity_comes_from_warm_jobs(monkeypatch):
    spec = importlib.util.spec_from_file_location("bench_serving", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    monkeypatch.setitem(sys.modules, "bench_serving", bench)
    spec.loader.exec_module(bench)
    from paper_2110_10156_gb300 import build
    build.build()
    from paper_2110_10156_gb300 import cs_ngf
    monkeypatch.setattr(cs_ngf, "Server", FakeServer)
    monkeypatch.setattr(bench, "serve_pair", lambda s: {k: np.zeros(s, np.float32) for k in ("A", "MA", "B", "MB")})
    args = argparse.Namespace(serve_jobs=2, serve_active=1, serve_batch=16, serve_policy="arrival", serve_load=0.7)
    m = bench.serving_measure(args)
    assert len(m["service_ms_per_rotation_alone"]) == len(bench.SERVE_SHAPES)
    assert all(v < 0.5 * 300.0 / 128 for v in m["service_ms_per_rotation_alone"].values())
