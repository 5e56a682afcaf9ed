"""The buffer of paths past their noise window only saves time: no call fails for want of its memory."""
from dataclasses import replace

import numpy as np
import pytest

import workloads as W
from paper_2410_13683_gb300 import fpt

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def _context(cap=1 << 16):
    ctx = fpt.fpt_init_model([replace(W.BM.model, max_steps=cap)])
    fpt.fpt_noise_table(ctx, 0, fpt.FPT_TABLE_USER_N, 16, 1.0, 0.0, 3.9, np.full(16, W.BM_S), np.zeros(16))
    return ctx


def _run(ctx, n, N=False):
    out = dict(nsteps=np.zeros(n, np.int32), logw=np.zeros(n), status=np.zeros(n, np.uint8))
    if N:
        out["N"] = np.zeros(n)
    fpt.fpt_run(ctx, [fpt.run_desc(0, n, seed=5, A=0.7)], [out])
    return out


@pytest.mark.parametrize("N", [False, True])
def test_a_call_that_needs_the_buffers_memory_gets_it(N):
    """200,000 paths hold 2.6 MB of results and 6.4 MB of buffer. A call of 400,000 (or one that asks for N, 1.6 MB)
    under a limit that leaves less than it needs; the same bits as without the limit, with graph replay and without."""
    require_gpu()
    n = 200000 if N else 400000
    with _context() as ctx:
        want = _run(ctx, n, N)
    for graph in (False, True):
        with _context() as ctx:
            fpt.fpt_set_launch(ctx, use_graph=graph)
            small = _run(ctx, 200000)
            used, _ = fpt.fpt_memory_in_use(ctx)
            fpt.fpt_set_memory_limit(ctx, used + (1 << 20))
            for _ in range(2):
                got = _run(ctx, n, N)
                for k in want:
                    np.testing.assert_array_equal(got[k], want[k])
            held, limit = fpt.fpt_memory_in_use(ctx)
            assert held <= limit
            # with the limit gone the next run has its buffer again
            fpt.fpt_set_memory_limit(ctx, 0)
            again = _run(ctx, 200000)
            for k in again:
                np.testing.assert_array_equal(again[k], small[k])
            assert fpt.fpt_memory_in_use(ctx)[0] >= held + 32 * 200000


@pytest.mark.parametrize("cap", [1 << 16, 4099])
def test_paths_that_find_the_buffer_full_go_on_in_the_stepper(cap):
    """A buffer of 1,000 paths, kept under a limit set afterwards, and 40,001 paths on one model."""
    require_gpu()
    n = 40001
    with _context(cap) as ctx:
        want = _run(ctx, n)
    with _context(cap) as ctx:
        fpt.fpt_set_memory_limit(ctx, 4 << 30)
        none = _run(ctx, n)
    with _context(cap) as ctx:
        _run(ctx, 1000)
        fpt.fpt_set_memory_limit(ctx, 4 << 30)
        full = _run(ctx, n)
    for k in want:
        np.testing.assert_array_equal(none[k], want[k])
        np.testing.assert_array_equal(full[k], want[k])
    assert (want["status"] == fpt.FPT_TRAJ_CAPPED).any() == (cap == 4099)
