"""The histogram kernels against the oracle's estimators at the edges of their classes, tiles and jackknife
blocks: bins narrower than a step, tails that cut a bin, the under- or the overflow, equal and zero weights."""
import numpy as np
import pytest

import workloads as W
from oracle import estimators as E
from paper_2410_13683_gb300 import fpt

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def _data(n, weights, seed=1):
    rng = np.random.default_rng(seed)
    N = rng.gamma(3.0, 2.0, n)
    lw = {"equal": np.full(n, -7.25), "zero": np.zeros(n), "wide": 150.0 * rng.standard_normal(n),
          "tilted": -0.3 * N + rng.standard_normal(n)}[weights]
    status = np.where(rng.random(n) < 0.01, fpt.FPT_TRAJ_CAPPED, fpt.FPT_TRAJ_PASSED)
    status[rng.random(n) < 0.01] = fpt.FPT_TRAJ_ABORTED
    return (N * 1e3).astype(np.int32), lw, status.astype(np.uint8)


@pytest.mark.parametrize("n, nb, lo, hi, tail, weights", [
    (1000, 1, 0.0, 40.0, 6.0, "tilted"),          # one class for every path
    (33, 64, 0.0, 20.0, 5.0, "tilted"),           # jackknife blocks of one or two paths
    (70001, 512, 0.5, 30.25, 8.3, "tilted"),      # a tail that cuts a bin; chunks that end inside a tile
    (200003, 1024, 0.0, 64.0, 0.2, "wide"),       # the largest count kept in shared memory; almost all in the tail
    (50001, 1025, 0.0, 64.0, 70.0, "tilted"),     # the first count beyond it; a tail above every bin
    (20000, 4096, 4.0, 4.25, 1.0, "zero"),        # bins of a sixteenth of a step; a tail that cuts the underflow
    (20000, 96, 1.0, 5.0, 9.0, "equal"),          # a tail that cuts the overflow
    (20000, 77, -3.0, 5.0, -1.0, "tilted"),       # a range that begins below zero, everything in the tail
])
def test_histogram_matches_the_oracle_at_the_edges(n, nb, lo, hi, tail, weights):
    torch = require_gpu()
    nst, lw, st = _data(n, weights)
    ref = E.histogram(nst, lw, st, 1e-3, lo, hi, nb)
    dev = [torch.from_numpy(x).cuda() for x in (nst, lw, st)]
    torch.cuda.synchronize()
    with fpt.fpt_init_model([W.BM.model]) as ctx:
        h = fpt.fpt_histogram_data(ctx, *dev, 1e-3, lo, hi, nb, N_tail=tail)
    assert np.array_equal(h["count"], ref.count)
    nz = ref.count > 0
    np.testing.assert_allclose(h["log_sum_w"][nz], ref.log_sum_w[nz], rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(h["log_sum_w2"][nz], ref.log_sum_w2[nz], rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(h["sum_lw"], ref.sum_lw, rtol=1e-12, atol=1e-9)
    with np.errstate(over="ignore", invalid="ignore"):
        P, se = E.p_weighted(ref)
    np.testing.assert_allclose(h["pdf"], P, rtol=1e-11)
    ok = np.isfinite(se)                          # the reference squares sums of up to e^600
    np.testing.assert_allclose(h["se_w"][ok], se[ok], rtol=1e-8, atol=1e-300)
    if weights != "wide":                         # a lognormal mean of e^(10^4) is beyond the reference
        Pl, _ = E.p_lognormal(ref)
        ok = np.isfinite(Pl)
        np.testing.assert_allclose(h["pdf_ln"][ok], Pl[ok], rtol=1e-9)
    assert (h["n_under"], h["n_over"], h["n_total"]) == (ref.n_under, ref.n_over, n)
    assert h["n_capped"] == np.count_nonzero(st == fpt.FPT_TRAJ_CAPPED)
    e, p, k = E.tail_ess(nst, lw, st, 1e-3, tail)
    assert h["n_tail"] == k
    assert h["ess_tail"] == pytest.approx(e, rel=1e-10)
    assert h["p_tail"] == pytest.approx(p, rel=1e-10)
    assert h["N_mean"] == pytest.approx(E.mean_N(nst, st, 1e-3), rel=1e-12)
    assert h["N_mean_w"] == pytest.approx(E.mean_N(nst, st, 1e-3, lw), rel=1e-10)
