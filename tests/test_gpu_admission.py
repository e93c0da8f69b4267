"""Stale-k admission, staleness histograms and the literal sliding-window
quantile rule on the GPU vs the oracle: kbar fp64 bits, admitted flags,
histogram counts, kappa, decisions and the window ring state all identical."""
import json
import os

import numpy as np
import pytest
import torch

import oracle
from pace_cases import DEV, as_np, assert_bits_equal, oracle_score, to_dev
from paper_2609_36830_gb300 import pace, workloads

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "hand_pool.json")


def _hand_arrays():
    h = json.load(open(GOLDEN))
    tr = h["trajectories"]
    tags = np.concatenate([np.array(t["tags"], np.int32) for t in tr])
    offsets = np.concatenate([[0], np.cumsum([len(t["tags"]) for t in tr])]).astype(np.int64)
    return tags, offsets, h["trainer_version"]


def _pools():
    out = [("hand",) + _hand_arrays()]
    for name, n in [("tiny", None), ("math7b", 512), ("multiturn", 480), ("sweep", 16384)]:
        p = workloads.make_pool(name, n_traj=n)
        out.append((name, p.tags, p.meta["offsets_host"], p.trainer_version))
    return out


@pytest.mark.parametrize("k_max", [0.0, 1.0, 2.5, 4.0, 8.0, 31.5])
def test_stale_k_matches_oracle(k_max):
    for name, tags, offsets, j in _pools():
        status = pace.new_status(DEV)
        kbar, adm = pace.stale_k(to_dev(tags), to_dev(offsets), j, k_max, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        st, okbar, oadm = oracle.stale_k(tags, offsets, j, k_max)
        assert st == 0
        assert_bits_equal(as_np(kbar), okbar, f"{name} kbar")
        np.testing.assert_array_equal(as_np(adm), oadm)


def test_stale_k_reports_tag_above_trainer_version():
    tags, offsets, j = _hand_arrays()
    status = pace.new_status(DEV)
    pace.stale_k(to_dev(tags), to_dev(offsets), j - 1, 1.0, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == pace.ERR_VERSION_ORDER


@pytest.mark.parametrize("n_bins,lo,hi", [(1, 0.0, 1.0), (7, 0.0, 8.0), (64, 0.5, 6.0),
                                          (4096, 0.0, 32.0)])
def test_histograms_match_oracle(n_bins, lo, hi):
    pool = workloads.make_pool("sweep", n_traj=16384)
    o = oracle_score(pool.tags, pool.meta["offsets_host"], pool.c_version, pool.s_pre,
                     pool.trainer_version, pool.window, group_size=8)
    U = pool.n_traj // 8
    _, _, _, k = oracle.budget(pool.n_traj, pool.n_target, 0.0, 0.9, 0.0, U)
    _, _, _, flags = oracle.select(o["unit_score"], 8, k)
    for key in ("kwait", "kgen", "score"):
        vals = o[key]
        hist = pace.staleness_histogram(to_dev(vals), to_dev(flags), lo, hi, n_bins)
        st, oh = oracle.histogram(vals, flags, lo, hi, n_bins)
        assert st == 0
        np.testing.assert_array_equal(as_np(hist).astype(np.uint32), oh)
    unit_flags = flags[::8].copy()
    hist = pace.staleness_histogram(to_dev(o["unit_score"]), to_dev(unit_flags), lo, hi, n_bins)
    _, oh = oracle.histogram(o["unit_score"], unit_flags, lo, hi, n_bins)
    np.testing.assert_array_equal(as_np(hist).astype(np.uint32), oh)


@pytest.mark.parametrize("capacity,batch,min_obs", [(512, 40, 32), (64, 0, 8), (4096, 100, 32)])
def test_quantile_admission_over_steps(capacity, batch, min_obs):
    """Five consecutive trainer steps, each on a fresh pool; both sides carry their own window."""
    gw = pace.ScoreWindow(capacity, DEV)
    ow = oracle.Window(capacity)
    for step in range(5):
        pool = workloads.make_pool("math7b", seed=7000 + step, n_traj=[512, 768, 384, 640, 512][step])
        o = oracle_score(pool.tags, pool.meta["offsets_host"], pool.c_version, pool.s_pre,
                         pool.trainer_version, pool.window, group_size=8)
        U = pool.n_traj // 8
        _, _, r_hat, _ = oracle.budget(pool.n_traj, pool.n_target, 0.5, 0.9, 0.1 * step, U)
        r_eff = min(r_hat, 0.9)
        status = pace.new_status(DEV)
        dec, kap = pace.quantile_admit(to_dev(o["unit_score"]), r_eff, batch, gw,
                                       min_obs=min_obs, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        st, odec, okap = oracle.quantile_admit(o["unit_score"], r_eff, batch, ow, min_obs=min_obs)
        assert st == 0
        assert float(kap.item()) == okap, step
        np.testing.assert_array_equal(as_np(dec), odec)
        state = as_np(gw.state)
        assert (int(state[0]), int(state[1])) == (ow.count, ow.head)
        np.testing.assert_array_equal(as_np(gw.values)[:ow.count], ow.values[:ow.count])


def test_quantile_admission_large_candidate_list():
    pool = workloads.make_pool("sweep", n_traj=131072 * 8 // 8)
    o = oracle_score(pool.tags, pool.meta["offsets_host"], pool.c_version, pool.s_pre,
                     pool.trainer_version, pool.window, group_size=8)
    gw, ow = pace.ScoreWindow(512, DEV), oracle.Window(512)
    for r, batch in [(0.0, 0), (0.5, 5000), (0.25, 0)]:
        dec, kap = pace.quantile_admit(to_dev(o["unit_score"]), r, batch, gw)
        torch.cuda.synchronize()
        _, odec, okap = oracle.quantile_admit(o["unit_score"], r, batch, ow)
        assert float(kap.item()) == okap
        np.testing.assert_array_equal(as_np(dec), odec)


@pytest.mark.parametrize("capacity,filled", [(1, 1), (5, 3), (512, 512), (513, 513),
                                             (4096, 4096), (4096, 2047), (64, 0)])
@pytest.mark.parametrize("n_cand,batch", [(1, 1), (33, 20), (1024, 0), (16384, 9000),
                                          (16385, 16384), (70001, 40000), (70001, 1), (0, 4)])
def test_quantile_admit_sizes(capacity, filled, n_cand, batch):
    """Window sizes around the values a thread holds, candidates around the 32 of a word
    and the 16,384 of a scan, batches that fill in an early chunk, on its edge or never;
    heavy ties and infinite scores.  Every output is exact."""
    rng = np.random.default_rng(capacity * 7 + n_cand)
    vals = rng.integers(0, 40, size=capacity) / 8.0
    vals[rng.random(capacity) < 0.02] = np.inf
    x = rng.integers(0, 40, size=n_cand) / 8.0
    head = int(rng.integers(0, capacity))
    if filled < capacity:
        head = max(head, filled) % capacity
    for r in (0.0, 1.0 / 3.0, 1.0):
        win = pace.ScoreWindow(capacity, DEV)
        win.values.copy_(to_dev(vals))
        win.state.copy_(torch.tensor([filled, head]))
        status = pace.new_status(DEV)
        dec, kappa = pace.quantile_admit(to_dev(x), r, batch, win, min_obs=2, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        recent = np.sort(vals[(head - filled + np.arange(filled)) % capacity])
        k = min(max(int(np.ceil((1.0 - r) * filled - 1e-9)), 1), max(filled, 1))
        okappa = recent[k - 1] if filled >= 2 else np.inf
        assert float(kappa.item()) == okappa
        keep = ~(x > okappa)
        before = np.cumsum(keep) - keep
        drawn = before < batch if batch > 0 else np.ones(n_cand, bool)
        np.testing.assert_array_equal(as_np(dec), np.where(drawn, keep, 2).astype(np.uint8))
        nd = int(drawn.sum())
        ring = vals.copy()
        for i in range(max(0, nd - capacity), nd):
            ring[(head + i) % capacity] = x[i]
        np.testing.assert_array_equal(as_np(win.values), ring)
        assert win.state.tolist() == [min(filled + nd, capacity), (head + nd) % capacity]


@pytest.mark.parametrize("lo,hi,n_bins", [(0.0, 32.0, 1000), (0.1, 0.7, 77), (-3.0, 1e-3, 4096),
                                          (0.0, 5e-324, 3), (-1e308, 1.5e308, 10),
                                          (1e-310, 1e-308, 50), (0.3, np.nextafter(0.3, 1), 2),
                                          (0.0, 10.0, 10), (0.0, 1e-280, 7), (0.0, 3e290, 9)])
def test_histogram_at_bin_edges(lo, hi, n_bins):
    """Values at every bin edge and a few ulps around it, on ranges up to the smallest and
    largest that doubles hold, where a shorter computation of the bin could go astray;
    counts exact (the oracle's division, product and floor)."""
    rng = np.random.default_rng(n_bins)
    with np.errstate(over="ignore", invalid="ignore"):
        e = lo + (hi - lo) * (np.arange(n_bins + 1) / n_bins)
        x = [rng.uniform(0, 1, 5000) * (hi / 2 - lo / 2) * 2 + lo]
    e = e[np.isfinite(e)]
    x += [e, np.array([lo, hi, np.inf, -np.inf])]
    for step in (1, 2, 3):
        y = e.copy()
        z = e.copy()
        for _ in range(step):
            y, z = np.nextafter(y, np.inf), np.nextafter(z, -np.inf)
        x += [y, z]
    x = np.concatenate(x)
    x = x[~np.isnan(x)]
    flags = (rng.random(x.size) < 0.5).astype(np.uint8)
    hist = pace.staleness_histogram(to_dev(x), to_dev(flags), lo, hi, n_bins)
    st, oh = oracle.histogram(x, flags, lo, hi, n_bins)
    assert st == 0
    np.testing.assert_array_equal(as_np(hist).astype(np.uint32), oh)


def test_histogram_where_the_width_overflows():
    """lo and hi are finite, hi - lo is not: x - lo overflows for the larger values below hi
    and their quotient is NaN.  They count in the first bin, none outside the histogram."""
    lo, hi, n_bins = -1e308, 1.5e308, 10
    x = np.array([0.9e308, 1.2e308, 1.49e308, -0.9e308, 0.0, 1.5e308, 1.7e308, -1.7e308])
    flags = np.array([0, 1, 0, 1, 0, 1, 0, 1], np.uint8)
    want = np.zeros((2, n_bins), np.uint32)
    want[0, [0, n_bins - 1]] = 3, 1
    want[1, [0, n_bins - 1]] = 3, 1
    hist = pace.staleness_histogram(to_dev(x), to_dev(flags), lo, hi, n_bins)
    np.testing.assert_array_equal(as_np(hist).astype(np.uint32), want)


@pytest.mark.parametrize("order", ["-+", "+-", "--", "++"])
@pytest.mark.parametrize("at", [(10, 11), (10, 40), (10, 590)])  # one warp, two, two passes
def test_kappa_of_both_zeros(at, order):
    """A threshold of zero is +0 where the window holds one, whichever thread has it, and
    -0 where every zero in it is."""
    zeros = {"-": -0.0, "+": 0.0}
    win = pace.ScoreWindow(600, DEV)
    vals = np.full(600, 5.0)
    vals[at[0]], vals[at[1]] = zeros[order[0]], zeros[order[1]]  # the two smallest
    win.values.copy_(to_dev(vals))
    win.state[0] = 600
    _, kappa = pace.quantile_admit(to_dev(np.ones(3)), 1.0 - 1.0 / 600, 0, win)
    got = as_np(kappa)[0]
    assert got == 0.0 and np.signbit(got) == ("+" not in order)
