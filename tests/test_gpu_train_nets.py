"""Training rounds of many networks: the networks that share a launch do not change each other's round."""
import numpy as np
import pytest

import workloads as W
from paper_2410_13683_gb300 import fpt
from paper_2410_13683_gb300 import train as TR

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count, capped", [(1, False), (16, False), (17, False), (17, True)])
def test_a_round_of_many_networks_equals_single_rounds(count, capped):
    """Counts around the networks of one launch (16), and one network to a launch under a memory limit, against
    each network's own round; bit for bit. The networks have different trajectory counts and clamps."""
    torch = require_gpu()
    S, Z = np.full(16, W.BM_S), np.zeros(16)
    kw = dict(segment=64, alpha_max=2.0)
    scale = (20.0, 100.0, 0.2)
    init = [fpt.canonical_params(W.mlp_init(40 + k, out_scale=0.2)) for k in range(count)]
    n = [64 + 37 * k for k in range(count)]
    adam = dict(lr=1e-3, step=1)
    with fpt.fpt_init_model([W.BM.model]) as ctx:
        fpt.fpt_noise_table(ctx, 0, fpt.FPT_TABLE_USER, 16, 1.0, -0.1, 0.2, S, Z)
        if capped:
            fpt.fpt_set_memory_limit(ctx, 8 << 30)
        props, P, B = TR.new_proposals(ctx, init, [(0.0,) * 3] * count, [scale] * count, **kw)
        m, v = torch.zeros_like(P), torch.zeros_like(P)
        torch.cuda.synchronize()
        stats = fpt.fpt_mlp_train_batch(ctx, [props[k].desc(0, n[k], seed=7, run_id=k) for k in range(count)], 0.5,
                                        [4.0] * count, adam, P, m, v, B)
    for k in range(count):
        with fpt.fpt_init_model([W.BM.model]) as ctx:
            fpt.fpt_noise_table(ctx, 0, fpt.FPT_TABLE_USER, 16, 1.0, -0.1, 0.2, S, Z)
            one = TR.new_proposal(ctx, init[k], (0.0,) * 3, scale, **kw)
            m1, v1 = torch.zeros_like(one.params), torch.zeros_like(one.params)
            torch.cuda.synchronize()
            st = fpt.fpt_mlp_train_round(ctx, one.desc(0, n[k], seed=7, run_id=k), n[k], 0.5, 4.0, adam, one.params,
                                         m1, v1, one.blob)
        for a, b in ((P[k], one.params), (m[k], m1), (v[k], v1), (B[k], one.blob)):
            assert torch.equal(a, b), k
        assert stats[k]["loss"] == st["loss"] and stats[k]["n_records"] == st["n_records"]
