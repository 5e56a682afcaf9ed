"""Trajectories that change warps in a launch's tail, in blocks that begin with several busy warps.

Launches of 40,001 paths on one block per SM: eight to sixteen warps of a block are busy when the tail begins, draw
their own normals, merge as paths end (or not: one network per run) and get helper warps when few are left. The same
paths 32 to a call are one warp that has a helper from its first group and never moves a lane. Bit for bit, for every
kind of lane state that moves: both Kahan pairs, the momentum's, the weights', windows and segment records."""
from dataclasses import replace

import numpy as np
import pytest

import workloads as W
from paper_2410_13683_gb300 import fpt
from paper_2410_13683_gb300 import train as TR

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

N = 40001
PARTS = list(range(0, 256, 32)) + [20000, 31111, N - 1]
KINDS = ("direct", "bias", "2d", "window", "models", "bump", "bump2d", "mlp", "nets", "mlp2d", "mlpbump")


def _run(ctx, runs):
    outs = [dict(nsteps=np.zeros(r.n_traj, np.int32), logw=np.zeros(r.n_traj), status=np.zeros(r.n_traj, np.uint8))
            for r in runs]
    fpt.fpt_run(ctx, runs, outs)
    return [np.concatenate([o[k] for o in outs]) for k in ("nsteps", "logw", "status")]


def _context(kind, cap):
    bump = "bump" in kind
    base = W.BUMP_MODEL if bump else W.BM.model
    ctx = fpt.fpt_init_model([replace(base, max_steps=cap)] * (2 if kind == "models" else 1))
    info = fpt.fpt_model_get_info(ctx, 0)
    lo, hi, amp = (info["phi_end"], info["phi_in"], 2e-6) if bump else (-0.1, 0.2, W.BM_S)
    S, Z = np.full(16, amp), np.zeros(16)
    for m in range(2 if kind == "models" else 1):
        if "2d" in kind:
            fpt.fpt_noise_table2(ctx, m, fpt.FPT_TABLE_USER2, 16, 1.0, lo, hi, (S, 0.1 * S, 0.2 * S))
        elif kind == "window":
            fpt.fpt_noise_table(ctx, m, fpt.FPT_TABLE_USER_N, 16, 1.0, 0.3, 4.0, S, Z)
        else:
            fpt.fpt_noise_table(ctx, m, fpt.FPT_TABLE_USER, 16, 1.0, lo, hi, S, 0.3 * S if bump else Z)
    return ctx


def _proposals(ctx, count=1):
    init = [fpt.canonical_params(W.mlp_init(14 + k, out_scale=0.3)) for k in range(count)]
    return TR.new_proposals(ctx, init, [(0.0, 0.0, 0.0)] * count, [(20.0, 100.0, 0.2)] * count, segment=64,
                            alpha_max=2.0)[0]


def _descs(kind, props, off, n):
    """The runs of paths off .. off + n: with several models or networks, the first and the second half of them."""
    two = kind in ("models", "nets")
    parts = [(0, off, n)] if not two else \
        [(0, off, max(0, min(n, N // 2 - off))), (1, max(off, N // 2), max(0, off + n - max(off, N // 2)))]
    runs = []
    for r, o, k in parts:
        model = r if kind == "models" else 0
        if props:
            runs.append(props[r].desc(model, k, seed=5, run_id=1 + r, traj_offset=o))
        else:
            A = 0.0 if kind == "direct" else 0.9
            runs.append(fpt.run_desc(model, k, seed=5, run_id=1 + r, A=A, A2=0.4 if "2d" in kind else 0.0, traj_offset=o))
    return runs


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("cap", [1 << 16, 5003])
def test_paths_end_alike_among_several_busy_warps_and_alone(kind, cap):
    require_gpu()
    with _context(kind, cap) as ctx:
        props = _proposals(ctx, 2 if kind == "nets" else 1) if kind in ("mlp", "nets", "mlp2d", "mlpbump") else None
        fpt.fpt_set_launch(ctx, block=512, blocks_per_sm=1, check_steps=32)
        whole = _run(ctx, _descs(kind, props, 0, N))
        assert (whole[0] > 0).all() and (whole[2] != fpt.FPT_TRAJ_ABORTED).all()
        assert len(np.unique(whole[0])) > 1
        for off in PARTS:
            part = _run(ctx, _descs(kind, props, off, min(32, N - off)))
            for a, b in zip(whole, part):
                np.testing.assert_array_equal(a[off:off + 32], b)


@pytest.mark.parametrize("kind", ["mlp", "mlp2d", "mlpbump"])
def test_segment_records_are_alike_among_several_busy_warps_and_alone(kind):
    require_gpu()
    cap = 1 << 13
    with _context(kind, cap) as ctx:
        prop = _proposals(ctx)[0]
        fpt.fpt_set_launch(ctx, block=512, blocks_per_sm=1, check_steps=32)
        whole = fpt.fpt_run_records(ctx, prop.desc(0, N, seed=5, run_id=1), cap=N * (cap // 64 + 1))
        assert whole["n_records"] == len(whole["unit"])
        for off in PARTS:
            k = min(32, N - off)
            part = fpt.fpt_run_records(ctx, prop.desc(0, k, seed=5, run_id=1, traj_offset=off))
            mine = (whole["unit"] >= off) & (whole["unit"] < off + k)
            assert mine.sum() == part["n_records"]
            for f in ("in", "tan", "raw", "sum_xi", "n0"):
                np.testing.assert_array_equal(whole[f][mine], part[f])
            np.testing.assert_array_equal(whole["unit"][mine] - off, part["unit"])
