"""The C-ABI library builds, loads without a GPU and exports every symbol that
include/*.h declares; its host-only budget function matches the oracle bit for
bit; host-side argument checks return before touching the device."""
import ctypes
import glob
import os
import re

import numpy as np
import pytest

import oracle
from paper_2609_36830_gb300 import build as pace_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def pace():
    pace_build.build()
    from paper_2609_36830_gb300 import pace as p
    p.lib()
    return p


def _declared_symbols():
    names = set()
    for h in glob.glob(os.path.join(ROOT, "include", "*.h")):
        txt = open(h).read()
        names.update(re.findall(r"PACE_API\s+[\w\s\*]+?\b(pace_\w+)\s*\(", txt))
    return names


def test_every_declared_symbol_is_exported(pace):
    declared = _declared_symbols()
    assert len(declared) >= 16
    L = ctypes.CDLL(pace.LIB_PATH)
    for name in sorted(declared):
        assert hasattr(L, name), name
    # the binding declares a signature for each of them
    assert declared == set(pace.SIGNATURES)


def test_status_strings_and_defaults(pace):
    assert pace.status_string(0) == "PACE_OK"
    assert pace.status_string(2) == "PACE_ERR_VERSION_ORDER"
    assert pace.status_string(99) == "PACE_ERR_UNKNOWN"
    assert pace.lib().pace_version() == 300  # 0.3.0: sharded selection, PaceLossArgs.partial
    sp = pace.PaceScoreParams()
    pace.lib().pace_score_params_default(ctypes.byref(sp))
    assert (sp.mode, sp.gamma, sp.min_obs, sp.group_size, sp.f_missing) == (0, 4, 32, 8, 1.0)
    bp = pace.PaceBudgetParams()
    pace.lib().pace_budget_params_default(ctypes.byref(bp))
    assert (bp.beta, bp.r_max, bp.r_hat_prev) == (0.0, 0.9, 0.0)
    lp = pace.PaceLossParams()
    pace.lib().pace_loss_params_default(ctypes.byref(lp))
    assert lp.eps_low == np.float32(0.2) and lp.eps_high == np.float32(0.28)
    assert lp.dual_clip == 10.0 and lp.agg == 0 and lp.std_unbiased == 1


def test_budget_matches_oracle_bitwise(pace):
    rng = np.random.default_rng(11)
    cases = [(47, 35, 0.0, 0.9, 0.0, 47), (64, 48, 0.0, 0.9, 0.0, 8), (6, 4, 0.5, 0.9, 0.2, 6),
             (100, 0, 0.0, 0.9, 0.0, 100), (10, 20, 0.3, 0.9, 0.5, 10)]
    for _ in range(3000):
        n = int(rng.integers(0, 3_000_000))
        g = int(rng.choice([1, 8, 12, 16]))
        cases.append((n, int(rng.integers(0, n + 2)), float(rng.choice([0.0, 0.3, 0.9, 0.99])),
                      float(rng.choice([0.9, 0.5, 1.0])), float(rng.random()), max(n // g, 0)))
    for n, nt, beta, rmax, prev, u in cases:
        st, r, rh, k = oracle.budget(n, nt, beta, rmax, prev, u)
        assert st == 0
        r2, rh2, k2 = pace.budget(n, u, pace.budget_params(nt, beta, rmax, prev))
        assert (r2, rh2, k2) == (r, rh, k), (n, nt, beta, rmax, prev, u)


def test_budget_rejects_bad_parameters(pace):
    with pytest.raises(pace.PaceError):
        pace.budget(10, 10, pace.budget_params(5, beta=1.0))
    with pytest.raises(pace.PaceError):
        pace.budget(10, 10, pace.budget_params(5, r_max=1.5))


def test_host_argument_checks_return_before_launch(pace):
    L = pace.lib()
    fake = ctypes.c_void_p(0x1000)
    p = pace.score_params(group_size=8)
    # 12 trajectories are not whole groups of 8
    st = L.pace_score_pool(fake, fake, fake, fake, 12, 100, 5, None, 0, ctypes.byref(p), None,
                           None, None, fake, None, fake, 1 << 20, None, None)
    assert st == pace.ERR_INVALID_ARG
    p = pace.score_params(gamma=0)
    st = L.pace_score_pool(fake, fake, fake, fake, 8, 100, 5, None, 0, ctypes.byref(p), None,
                           None, None, fake, None, fake, 1 << 20, None, None)
    assert st == pace.ERR_INVALID_ARG
    p = pace.score_params()
    st = L.pace_score_pool(fake, fake, fake, fake, 8, 100, 5, fake, 5000, ctypes.byref(p), None,
                           None, None, fake, None, fake, 1 << 20, None, None)
    assert st == pace.ERR_UNSUPPORTED_SHAPE  # window longer than 4096
    st = L.pace_select_k(fake, 10, 1, 11, fake, fake, None, fake, 1 << 20, None, None)
    assert st == pace.ERR_INVALID_ARG  # k > U
    b = pace.PaceBatch(fake, None, None, 4, 100)
    st = L.pace_token_logprob(ctypes.byref(b), fake, fake, fake, 100, 1000, 1.0, fake, None,
                              None, fake, 1 << 20, None, None)
    assert st == pace.ERR_UNSUPPORTED_SHAPE  # hidden size not a multiple of 64
    st = L.pace_token_logprob(ctypes.byref(b), fake, fake, fake, 128, 1000, 0.0, fake, None,
                              None, fake, 1 << 20, None, None)
    assert st == pace.ERR_INVALID_ARG  # temperature must be > 0
    # the LM head reads the rows in the loss by index: no copy of the hidden rows
    # in the workspace, so its size does not depend on the hidden size
    ws = L.pace_token_logprob_workspace_size(1000, 10, 128, 1000)
    assert 1000 * 4 < ws < 1000 * 128 * 2
    assert L.pace_token_logprob_workspace_size(1000, 10, 16384, 1000) == ws
    assert L.pace_score_pool_workspace_size(1000, 512) >= 16 * 1000


def test_lmhead_split_control_range(pace):
    L = pace.lib()
    for bad in (-1, 9, 1 << 20):
        assert L.pace_set_lmhead_splits(bad) == pace.ERR_INVALID_ARG
    for good in (0, 1, 2, 4, 8):
        assert L.pace_set_lmhead_splits(good) == pace.OK
    assert L.pace_set_lmhead_splits(0) == pace.OK  # back to the automatic choice


def test_score_fusion_control_range(pace):
    L = pace.lib()
    assert L.pace_set_score_fused_min_traj(-1) == pace.ERR_INVALID_ARG
    for good in (0, 1, 1 << 18, 1 << 62):
        assert L.pace_set_score_fused_min_traj(good) == pace.OK
    assert L.pace_score_fused_min_traj_default() == 1 << 18
    pace.set_score_fused_min_traj()


def test_shard_selection_argument_checks_return_before_launch(pace):
    """The sharded rejection's calls refuse bad arguments on the host, before any launch."""
    L = pace.lib()
    fake = ctypes.c_void_p(0x1000)
    ws = ctypes.c_void_p(0x100000)  # 256-byte aligned, never dereferenced here
    n = 1 << 20
    assert L.pace_select_shard_workspace_size(100) > 0
    assert L.pace_select_shard_workspace_size(-1) == 0
    # pass out of range, a negative k, a missing histogram, no previous histogram after pass 0
    assert L.pace_select_shard_pass(fake, 100, 6, 3, fake, fake, ws, n, None, None) == \
        pace.ERR_INVALID_ARG
    assert L.pace_select_shard_pass(fake, 100, 0, -1, None, fake, ws, n, None, None) == \
        pace.ERR_INVALID_ARG
    assert L.pace_select_shard_pass(fake, 100, 0, 3, None, None, ws, n, None, None) == \
        pace.ERR_INVALID_ARG
    assert L.pace_select_shard_pass(fake, 100, 2, 3, None, fake, ws, n, None, None) == \
        pace.ERR_INVALID_ARG
    # workspace missing, unaligned or too small
    assert L.pace_select_shard_pass(fake, 100, 0, 3, None, fake, None, n, None, None) == \
        pace.ERR_WORKSPACE
    assert L.pace_select_shard_pass(fake, 100, 0, 3, None, fake, ctypes.c_void_p(0x100008), n,
                                    None, None) == pace.ERR_WORKSPACE
    assert L.pace_select_shard_pass(fake, 100, 0, 3, None, fake, ws, 8, None, None) == \
        pace.ERR_WORKSPACE
    # ties: missing output; write: ids past int32, missing tie count, bad group size
    assert L.pace_select_shard_ties(fake, 100, fake, None, ws, n, None, None) == \
        pace.ERR_INVALID_ARG
    assert L.pace_select_shard_write(fake, 100, 8, 3, fake, (1 << 31) - 100, fake, fake, fake,
                                     None, ws, n, None, None) == pace.ERR_INVALID_ARG
    assert L.pace_select_shard_write(fake, 100, 8, 3, None, 0, fake, fake, fake, None, ws, n,
                                     None, None) == pace.ERR_INVALID_ARG
    assert L.pace_select_shard_write(fake, 100, 0, 3, fake, 0, fake, fake, fake, None, ws, n,
                                     None, None) == pace.ERR_INVALID_ARG
    assert L.pace_loss_from_partial(None, fake, None) == pace.ERR_INVALID_ARG
    assert L.pace_div_selftest(None, None, -1, None, None, None, None, None) == \
        pace.ERR_INVALID_ARG


def test_workspaces_never_shrink_as_batches_grow(pace):
    """A workspace made for the largest batch serves every smaller one: no size query falls
    as rows, sequences, trajectories or units grow, around every multiple at which the row
    walk's launches change shape and at each power of two."""
    L = pace.lib()
    step = 256 * 8 * 456  # rows of one tile a warp in a full launch
    rows = sorted({max(0, k * r + d) for k in (1, 2, 3) for d in (-1, 0, 1, 255, 256, 257, 4096)
                   for r in (step, step // 2, 16384, 32768)}
                  | {max(0, 2 ** e + d) for e in range(0, 23) for d in (-1, 0, 1)}
                  | {610_000, 1_000_000, 1_200_000, 5_400_000})
    seqs = [0, 1, 7, 8, 9, 64, 1000, 1024, 100_000]
    heads = ((64, 64), (256, 2048), (64, 4033), (1024, 50_001), (3584, 152_064))

    def nondecreasing(f, xs):
        sizes = [f(x) for x in xs]
        assert all(a <= b for a, b in zip(sizes, sizes[1:])), \
            [(x, a, b) for x, a, b in zip(xs, sizes, sizes[1:]) if a > b][:3]

    for f in (L.pace_surrogate_loss_workspace_size, L.pace_surrogate_backward_workspace_size):
        for s in seqs:
            nondecreasing(lambda n: f(n, s), rows)
        for n in rows[::5]:
            nondecreasing(lambda s: f(n, s), seqs)
    for f in (L.pace_token_logprob_workspace_size, L.pace_prefix_score_workspace_size,
              L.pace_token_logprob_backward_workspace_size):
        for H, V in heads:
            for s in (1, 1024):
                nondecreasing(lambda n: f(n, s, H, V), rows)
            for n in rows[::9]:
                nondecreasing(lambda s: f(n, s, H, V), seqs)
    for w in (0, 1, 512, 4096):
        nondecreasing(lambda n: L.pace_score_pool_workspace_size(n, w), rows)
    for n in rows[::5]:
        nondecreasing(lambda w: L.pace_score_pool_workspace_size(n, w), [0, 1, 511, 512, 4096])
    nondecreasing(L.pace_stale_k_workspace_size, rows)
    nondecreasing(L.pace_select_workspace_size, rows)
    nondecreasing(L.pace_select_shard_workspace_size, rows)


@pytest.mark.parametrize("n,H,V,parts", [(16384, 256, 2048, 0), (65536, 64, 4032, 0),
                                         (16384, 1024, 4033, 2), (2582, 2048, 12288, 6),
                                         (2582, 2048, 151936, 8)])
def test_backward_workspace_holds_what_the_vocabulary_needs(pace, n, H, V, parts):
    """Gathered rows, one chunk of G, and dH's partial tiles: at most 75 tiles of 256 x 256
    floats in `parts` parts, one per 32 K steps of 64 vocabulary entries and at most 8, none
    where that is below 2; the rest (row lists, log-prob partials) is below 128 bytes a row
    and 1 MB."""
    chunk = min(n, 32768)
    chunk = (chunk + 127) // 128 * 128
    tiles = min((chunk + 255) // 256 * ((H + 255) // 256), 75)
    need = 2 * n * H + 2 * chunk * ((V + 63) // 64 * 64) + tiles * parts * 256 * 256 * 4
    got = pace.lib().pace_token_logprob_backward_workspace_size(n, 8, H, V)
    assert need <= got <= need + 128 * n + (1 << 20)
