"""Histograms of weights that are zero (ln w = -inf), infinite, not a number or masked by the type's lowest value:
each spoils what it is part of and nothing else."""
import numpy as np
import pytest

import workloads as W
from oracle import estimators as E
from paper_2410_13683_gb300 import fpt

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

N, LO, HI, NB, TAIL = 30011, 1.0, 9.0, 64, 6.05      # bins of 125 steps; the tail cuts bin 40 (6.0 to 6.125)
LOWEST = -np.finfo(np.float64).max


def _data(case):
    rng = np.random.default_rng(3)
    t = rng.gamma(3.0, 1.6, N)
    nst = (t * 1e3).astype(np.int32)
    lw = -0.3 * t + rng.standard_normal(N)
    st = np.where(rng.random(N) < 0.01, fpt.FPT_TRAJ_CAPPED, fpt.FPT_TRAJ_PASSED).astype(np.uint8)
    T = nst.astype(np.float64) * 1e-3
    b = np.floor((T - LO) / ((HI - LO) / NB)).astype(np.int64)
    some = rng.random(N) < 0.03
    where = {"some": some, "lowest": some, "bins": (b == 5) | (b == 6), "under": T < LO, "over": T >= HI,
             "cut, above": (b == 40) & (T >= TAIL), "cut, below": (b == 40) & (T < TAIL), "cut": b == 40,
             "cut, some": (b == 40) & some, "tail": T >= TAIL, "all": T >= 0.0, "bin of the tail": b == 50,
             "infinite": (b == 20) & some, "infinite in the tail": (b == 50) & some, "infinite and zero": b == 20,
             "nan": (b == 20) & some, "nan in the tail": (b == 50) & some}[case]
    v = {"lowest": LOWEST, "infinite": np.inf, "infinite in the tail": np.inf, "infinite and zero": np.inf,
         "nan": np.nan, "nan in the tail": np.nan}.get(case, -np.inf)
    lw[where] = v
    if case == "infinite and zero":
        lw[np.flatnonzero(where)[::2]] = -np.inf
    assert (where & (st == 0)).any()
    return nst, lw, st


CASES = ["some", "lowest", "bins", "under", "over", "cut, above", "cut, below", "cut", "cut, some", "tail", "all",
         "bin of the tail", "infinite", "infinite in the tail", "infinite and zero", "nan", "nan in the tail"]


@pytest.mark.parametrize("data", [True, False])
@pytest.mark.parametrize("case", CASES)
@pytest.mark.filterwarnings("ignore::RuntimeWarning")
def test_a_weight_spoils_only_what_it_is_part_of(case, data):
    torch = require_gpu()
    nst, lw, st = _data(case)
    ref = E.histogram(nst, lw, st, 1e-3, LO, HI, NB)
    dev = [torch.from_numpy(x).cuda() for x in (nst, lw, st)]
    torch.cuda.synchronize()
    if data:
        with fpt.fpt_init_model([W.BM.model]) as ctx:
            h = fpt.fpt_histogram_data(ctx, *dev, 1e-3, LO, HI, NB, N_tail=TAIL)
    else:
        out = torch.zeros(fpt.hist_out_doubles(NB), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        fpt.fpt_histogram_noalloc(*dev, 1e-3, LO, HI, NB, out, N_tail=TAIL)
        torch.cuda.synchronize()
        h = fpt.unpack_hist(out.cpu().numpy(), NB)
    assert np.array_equal(h["count"], ref.count)
    np.testing.assert_allclose(h["log_sum_w"], ref.log_sum_w, rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(h["log_sum_w2"], ref.log_sum_w2, rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(h["sum_lw"], ref.sum_lw, rtol=1e-12, atol=1e-9)
    np.testing.assert_allclose(h["sum_lw2"], ref.sum_lw2, rtol=1e-12, atol=1e-9)
    P, _ = E.p_weighted(ref)
    np.testing.assert_allclose(h["pdf"], P, rtol=1e-11)
    fine = np.isfinite(ref.log_sum_w)
    np.testing.assert_allclose(h["se_w"][fine], E.p_weighted(ref)[1][fine], rtol=1e-8, atol=1e-300)
    np.testing.assert_allclose(h["se_jk"][fine], E.p_jackknife(ref)[1][fine], rtol=1e-8, atol=1e-300)
    # the lognormal mean of sums that are not finite: the variance counts as zero, but
    # is infinite where only the sum of squares is (a mask of the type's lowest value)
    m = ref.sum_lw / ref.count
    s2 = np.fmax((ref.sum_lw2 - ref.count * m * m) / (ref.count - 1), 0.0)
    s2[np.isfinite(ref.sum_lw) & np.isinf(ref.sum_lw2)] = np.inf
    want = ref.count / N * np.exp(m + 0.5 * s2) / ref.db
    odd = ~np.isfinite(ref.sum_lw2) & (ref.count >= 2)
    np.testing.assert_array_equal(h["pdf_ln"][odd], want[odd])
    np.testing.assert_allclose(h["pdf_ln"][~odd], want[~odd], rtol=1e-9)
    # the scalars
    assert (h["n_under"], h["n_over"], h["n_total"]) == (ref.n_under, ref.n_over, N)
    p = st == fpt.FPT_TRAJ_PASSED
    T, l = nst[p].astype(np.float64) * 1e-3, lw[p]
    assert h["N_mean"] == pytest.approx(T.mean(), rel=1e-12)
    w = np.exp(l - l.max())
    sw, swn = w.sum(), (w * T).sum()
    assert h["N_mean_w"] == pytest.approx(swn / sw if sw > 0 else np.nan, rel=1e-10, nan_ok=True)
    tail = T >= TAIL
    mt = l[tail].max()
    wt = np.exp(l[tail] - mt)
    assert h["n_tail"] == tail.sum()
    assert h["ess_tail"] == pytest.approx(wt.sum() ** 2 / (wt * wt).sum() if (wt * wt).sum() > 0 else 0.0, rel=1e-10)
    assert h["p_tail"] == pytest.approx(np.exp(mt + np.log(wt.sum())) / N if wt.sum() > 0 else 0.0, rel=1e-10)
    np.testing.assert_equal(h["log_max_w"], l.max())
