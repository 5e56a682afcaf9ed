"""The launch's tail: trajectories that move between warps, refill or end in any interval give the results
they give alone."""
from dataclasses import replace

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

fpt = pytest.importorskip("paper_2410_13683_gb300.fpt")


def _run(ctx, runs):
    outs = [dict(nsteps=np.zeros(r.n_traj, np.int32), logw=np.zeros(r.n_traj), status=np.zeros(r.n_traj, np.uint8))
            for r in runs]
    fpt.fpt_run(ctx, runs, outs)
    return [np.concatenate([o[k] for o in outs]) for k in ("nsteps", "logw", "status")]


def _context(kind, cap):
    ctx = fpt.fpt_init_model([replace(W.BM.model, max_steps=cap)])
    S, Z = np.full(16, W.BM_S), np.zeros(16)
    if kind == "2d":
        fpt.fpt_noise_table2(ctx, 0, fpt.FPT_TABLE_USER2, 16, 1.0, -0.1, 0.2, (S, 0.1 * S, 0.2 * S))
    elif kind == "window":
        fpt.fpt_noise_table(ctx, 0, fpt.FPT_TABLE_USER_N, 16, 1.0, 0.3, 4.0, S, Z)
    else:
        fpt.fpt_noise_table(ctx, 0, fpt.FPT_TABLE_USER, 16, 1.0, -0.1, 0.2, S, Z)
    return ctx


@pytest.mark.parametrize("kind", ["bias", "2d", "window", "mlp"])
@pytest.mark.parametrize("cap", [1 << 16, 5003, 5120, 2])
def test_results_do_not_depend_on_the_company_of_a_path(kind, cap):
    """n paths in one launch (warps with idle lanes, blocks that merge their last lanes) against the same
    paths 32 to a call, where no lane can move; bit for bit. The caps fall on, inside and before an interval."""
    n = 4097
    with _context(kind, cap) as ctx:
        def desc(off, k):
            if kind == "mlp":
                return prop.desc(0, k, seed=5, run_id=1, traj_offset=off)
            return fpt.run_desc(0, k, seed=5, run_id=1, A=0.9, A2=0.4 if kind == "2d" else 0.0, traj_offset=off)

        if kind == "mlp":
            from paper_2410_13683_gb300 import train as TR
            prop = TR.new_proposal(ctx, fpt.canonical_params(W.mlp_init(14, out_scale=0.3)), shift=(0.0, 0.0, 0.0),
                                   scale=(20.0, 100.0, 0.2), segment=64, alpha_max=2.0)
        whole = _run(ctx, [desc(0, n)])
        for off in list(range(0, 512, 32)) + [4064, 4096]:
            part = _run(ctx, [desc(off, min(32, n - off))])
            for a, b in zip(whole, part):
                np.testing.assert_array_equal(a[off:off + 32], b)
        assert (whole[0][whole[2] == fpt.FPT_TRAJ_CAPPED] == cap).all()


@pytest.mark.parametrize("n", [1, 31, 33, 511, 513, 152 * 1024 + 1])
def test_every_path_runs_once_at_the_edges_of_a_launch(n):
    """Counts around a warp, a block and the resident lanes: each path has a result, equal to that of the
    same ids in two runs of one call."""
    with _context("bias", 6000) as ctx:
        a = _run(ctx, [fpt.run_desc(0, n, seed=6, A=0.5)])
        k = n // 2
        b = _run(ctx, [fpt.run_desc(0, k, seed=6, A=0.5), fpt.run_desc(0, n - k, seed=6, A=0.5, traj_offset=k)])
        for x, y in zip(a, b):
            np.testing.assert_array_equal(x, y)
        assert (a[0] > 0).all() and (a[2] != fpt.FPT_TRAJ_ABORTED).all()


@pytest.mark.parametrize("cap", [1 << 16, 4099])
def test_paths_past_their_window_end_alike_with_and_without_the_buffer(cap):
    """Paths that outlive their noise window are finished by a kernel of their own; where the context's memory
    is capped the stepper takes those steps itself. Bit for bit, beside a run whose window never ends."""
    S, Z = np.full(16, W.BM_S), np.zeros(16)
    got = []
    for capped in (False, True):
        models = [replace(W.BM.model, max_steps=cap)] * 2
        with fpt.fpt_init_model(models) as ctx:
            fpt.fpt_noise_table(ctx, 0, fpt.FPT_TABLE_USER_N, 16, 1.0, 0.0, 3.9, S, Z)
            fpt.fpt_noise_table(ctx, 1, fpt.FPT_TABLE_USER_N, 16, 1.0, 0.5, 90.0, S, Z)
            if capped:
                fpt.fpt_set_memory_limit(ctx, 4 << 30)
            got.append(_run(ctx, [fpt.run_desc(0, 3001, seed=5, A=0.7),
                                  fpt.run_desc(1, 1501, seed=5, run_id=1, A=0.7)]))
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
