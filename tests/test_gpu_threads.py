"""Contexts on host threads of their own that launch the same kernels with different amounts of shared memory."""
import threading
from dataclasses import replace

import numpy as np
import pytest

import workloads as W
from paper_2410_13683_gb300 import fpt

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

ROUNDS = 2000


def _both(*works):
    """Runs the works on a thread each, ROUNDS times; their errors."""
    errors, gate = [], threading.Barrier(len(works))

    def loop(work):
        try:
            gate.wait()
            for _ in range(ROUNDS):
                work()
        except Exception as e:          # noqa: BLE001 -- reported by the test
            errors.append(e)

    threads = [threading.Thread(target=loop, args=(w,)) for w in works]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


def _context(points):
    ctx = fpt.fpt_init_model([replace(W.BM.model, max_steps=4)])
    fpt.fpt_noise_table(ctx, 0, fpt.FPT_TABLE_USER, points, 1.0, -0.1, 0.2, np.full(points, W.BM_S), np.zeros(points))
    fpt.fpt_set_launch(ctx, use_graph=False)
    return ctx


def test_launches_of_several_threads_do_not_refuse_each_other():
    """Tables of 16 and of 8,192 points (0.3 and 131 KB), each staged in shared memory by the same kernel."""
    require_gpu()
    with _context(16) as a, _context(8192) as b, _context(16) as c, _context(8192) as d:
        runs = [fpt.run_desc(0, 64, seed=3, A=0.5)]
        assert not _both(*[lambda ctx=ctx: fpt.fpt_run(ctx, runs) for ctx in (a, b, c, d)])
        got = []
        for ctx in (a, b, c, d):
            out = [dict(nsteps=np.zeros(64, np.int32), logw=np.zeros(64))]
            fpt.fpt_run(ctx, runs, out)
            got.append(out[0]["logw"])
        np.testing.assert_array_equal(got[0], got[2])
        np.testing.assert_array_equal(got[1], got[3])


def test_histograms_of_several_threads_do_not_refuse_each_other():
    """512, 1,024 and 4,096 bins: 80 to 141 KB of shared memory in the summing kernel."""
    require_gpu()
    rng = np.random.default_rng(2)
    nst, lw, st = rng.integers(1, 9000, 5000, dtype=np.int32), rng.normal(size=5000), np.zeros(5000, np.uint8)
    with _context(16) as a, _context(16) as b, _context(16) as c:
        def work(ctx, bins):
            h = fpt.fpt_histogram_data(ctx, nst, lw, st, 1e-3, 0.0, 9.0, bins)
            assert h["count"].sum() == 5000

        assert not _both(lambda: work(a, 512), lambda: work(b, 1024), lambda: work(c, 4096))
