"""GRPO advantages and the clipped surrogate on the GPU vs the oracle.

Advantages are fp64 on both sides and rounded to float32 once: bit-identical.
The surrogate's per-token terms are fp32 on the GPU and fp64 in the oracle;
the loss must agree within 1e-3 relative (observed ~1e-7) and the ratios
within 1e-5 relative.  Inputs here are seeded synthetic log-probs, so the
oracle computes the full loss even at the largest batch sizes."""
import numpy as np
import pytest
import torch

import oracle
from pace_cases import DEV, as_np, to_dev
from paper_2609_36830_gb300 import pace, workloads

pytestmark = pytest.mark.gpu


def test_advantages_of_few_and_of_many_groups_cost_alike():
    """Whatever the number of groups, the time per group does not grow with it: lanes per
    group repeat its fp64 sums, so they may not be used where throughput counts (1M
    sequences in groups of 32 took 198 us that way, 47 with a thread per group)."""
    n, G = 1 << 20, 32
    r, out = torch.rand(n, device=DEV), torch.empty(n, device=DEV)
    times = []
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            pace.group_advantages(r, G, out=out)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) / 20)
    assert min(times) < 0.1  # ms


# the last four: around the number of groups from which a thread takes each
@pytest.mark.parametrize("G,n_seq,p_acc", [(8, 64, 1.0), (8, 512, 0.75), (12, 1200, 0.5),
                                           (1, 300, 0.8), (16, 16, 0.3), (2, 12288, 0.6),
                                           (2, 12290, 0.6), (12, 49152, 0.6), (12, 49164, 0.6)])
@pytest.mark.parametrize("unbiased", [True, False])
def test_advantages_bitwise(G, n_seq, p_acc, unbiased):
    rng = np.random.default_rng(G * 1000 + n_seq)
    r = (rng.random(n_seq) < 0.4).astype(np.float32)
    r[: G] = 1.0  # an all-equal group
    acc = (rng.random(n_seq) < p_acc).astype(np.uint8)
    eps = np.float32(1e-6)
    adv = pace.group_advantages(to_dev(r), G, seq_accepted=to_dev(acc), adv_eps=eps,
                                std_unbiased=unbiased)
    st, oadv = oracle.group_advantages(r, G, seq_accepted=acc, eps=float(eps), unbiased=unbiased)
    assert st == 0
    np.testing.assert_array_equal(as_np(adv), oadv.astype(np.float32))


@pytest.mark.parametrize("G,groups", [(8, 6144), (8, 6145), (32, 2049), (1, 9000), (40, 300)])
@pytest.mark.parametrize("call", ["derivative", "few rows", "rows"])
def test_advantages_in_other_launches(G, groups, call):
    """The advantages that the count's or the list's launch computes in its extra blocks, on
    both sides of the number of groups from which a thread takes each, have the bits of a
    launch of their own."""
    rng = np.random.default_rng(G + groups)
    n_seq = G * groups
    n = {"derivative": 20_000, "few rows": 3000, "rows": 20_000}[call]
    so = np.sort(rng.integers(0, n + 1, size=n_seq + 1)).astype(np.int64)
    so[0], so[-1] = 0, n
    acc = to_dev((rng.random(n_seq) < 0.7).astype(np.uint8))
    reward = to_dev(rng.random(n_seq).astype(np.float32))
    want = as_np(pace.group_advantages(reward, G, seq_accepted=acc))
    adv = torch.full((n_seq,), 7.0, device=DEV)
    la = pace.make_loss_args(torch.zeros(n, device=DEV), reward, G, pace.loss_params(),
                             torch.zeros(1, dtype=torch.float64, device=DEV), adv_out=adv)
    b = pace.make_batch(to_dev(so), n, seq_accepted=acc)
    if call == "derivative":
        pace.surrogate_backward(b, torch.zeros(n, device=DEV), la)
    else:
        hidden = torch.zeros((n, 64), dtype=torch.bfloat16, device=DEV)
        pace.token_logprob(b, hidden, hidden[:64], torch.zeros(n, dtype=torch.int32, device=DEV),
                           loss=la)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(as_np(adv), want)


def _batch(rows, seed, accept_p=0.75):
    pool = workloads.make_pool(*rows)
    rw = workloads.make_rows(pool)
    rng = np.random.default_rng(seed)
    lp = (workloads.uniform_center(pool.spec.vocab or 1000)
          + rng.standard_normal(rw.n_rows)).astype(np.float32)
    behav = workloads.behaviour_logprob(rw, pool.trainer_version,
                                        workloads.uniform_center(pool.spec.vocab or 1000), seed)
    acc = (rng.random(pool.n_traj) < accept_p).astype(np.uint8)
    return pool, rw, lp, behav, acc


@pytest.mark.parametrize("rows", [("tiny", None), ("math7b", 512), ("multiturn", 480),
                                  ("moe", None)])
@pytest.mark.parametrize("agg", [pace.AGG_TOKEN_MEAN, pace.AGG_SEQ_MEAN_TOKEN_MEAN])
def test_surrogate_matches_oracle(rows, agg):
    pool, rw, lp, behav, acc = _batch(rows, 3)
    params = pace.loss_params(eps_low=pool.spec.eps_low, eps_high=pool.spec.eps_high,
                              agg=agg)
    loss = torch.zeros(1, dtype=torch.float64, device=DEV)
    ratio = torch.empty(rw.n_rows, dtype=torch.float32, device=DEV)
    adv = torch.empty(pool.n_traj, dtype=torch.float32, device=DEV)
    la = pace.make_loss_args(to_dev(behav), to_dev(pool.reward), pool.group_size, params, loss,
                             adv_out=adv, ratio_out=ratio)
    b = pace.make_batch(to_dev(rw.row_offsets), rw.n_rows, seq_accepted=to_dev(acc),
                        mask=to_dev(rw.mask))
    status = pace.new_status(DEV)
    pace.surrogate_loss(b, to_dev(lp), la, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    st, oadv = oracle.group_advantages(pool.reward, pool.group_size, seq_accepted=acc,
                                       eps=float(np.float32(1e-6)))
    np.testing.assert_array_equal(as_np(adv), oadv.astype(np.float32))
    st, oloss, oratio, _ = oracle.surrogate(lp, behav, rw.row_offsets, oadv,
                                            mask=rw.mask, seq_accepted=acc,
                                            eps_low=float(np.float32(pool.spec.eps_low)),
                                            eps_high=float(np.float32(pool.spec.eps_high)),
                                            dual_clip=10.0, agg=agg)
    assert st == 0
    gl = float(loss.item())
    assert abs(gl - oloss) <= 1e-3 * max(abs(oloss), 1e-12), (gl, oloss)
    np.testing.assert_allclose(as_np(ratio), oratio, rtol=1e-5, atol=0)


def test_on_policy_identity_on_gpu():
    pool, rw, lp, _, acc = _batch(("tiny", None), 9, accept_p=1.0)
    loss = torch.zeros(1, dtype=torch.float64, device=DEV)
    ratio = torch.empty(rw.n_rows, dtype=torch.float32, device=DEV)
    adv = torch.empty(pool.n_traj, dtype=torch.float32, device=DEV)
    la = pace.make_loss_args(to_dev(lp), to_dev(pool.reward), pool.group_size,
                             pace.loss_params(), loss, adv_out=adv, ratio_out=ratio)
    b = pace.make_batch(to_dev(rw.row_offsets), rw.n_rows, mask=to_dev(rw.mask))
    pace.surrogate_loss(b, to_dev(lp), la)
    torch.cuda.synchronize()
    r = as_np(ratio)[rw.mask.astype(bool)]
    assert (r == 1.0).all()
    st, oadv = oracle.group_advantages(pool.reward, pool.group_size, eps=float(np.float32(1e-6)))
    a_row = np.repeat(oadv, np.diff(rw.row_offsets))[rw.mask.astype(bool)]
    expect = -a_row.sum() / a_row.size
    assert abs(float(loss.item()) - expect) <= 1e-9 + 1e-6 * abs(expect)


def test_empty_loss_is_zero_and_bad_offsets_reported():
    so = np.array([0, 3, 5], np.int64)
    loss = torch.full((1,), 7.0, dtype=torch.float64, device=DEV)
    la = pace.make_loss_args(to_dev(np.zeros(5, np.float32)), to_dev(np.ones(2, np.float32)), 2,
                             pace.loss_params(), loss)
    b = pace.make_batch(to_dev(so), 5, mask=to_dev(np.zeros(5, np.uint8)))
    pace.surrogate_loss(b, to_dev(np.zeros(5, np.float32)), la)
    torch.cuda.synchronize()
    assert float(loss.item()) == 0.0
    bad = np.array([0, 4, 3], np.int64)
    b = pace.make_batch(to_dev(bad), 5)
    status = pace.new_status(DEV)
    pace.surrogate_loss(b, to_dev(np.zeros(5, np.float32)), la, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == pace.ERR_INVALID_ARG


@pytest.mark.parametrize("call", ["logprob", "logprob_with_loss", "prefix", "loss", "derivative"])
def test_bad_offsets_of_an_empty_batch_reported(call):
    """No rows, offsets that name some: every call says so."""
    b = pace.make_batch(to_dev(np.array([0, 2, 5, 9], np.int64)), 0)
    status = pace.new_status(DEV)
    hidden = torch.empty(0, 64, dtype=torch.bfloat16, device=DEV)
    w = torch.zeros(64, 64, dtype=torch.bfloat16, device=DEV)
    y = torch.empty(0, dtype=torch.int32, device=DEV)
    empty = torch.empty(0, device=DEV)
    loss = torch.full((1,), 7.0, dtype=torch.float64, device=DEV)
    la = pace.make_loss_args(torch.zeros(1, device=DEV), to_dev(np.ones(3, np.float32)), 3,
                             pace.loss_params(), loss)
    if call == "prefix":
        pace.prefix_score(b, hidden, w, y, torch.zeros(1, device=DEV), status=status)
    elif call == "loss":
        pace.surrogate_loss(b, empty, la, status=status)
    elif call == "derivative":
        pace.surrogate_backward(b, empty, la, status=status)
    else:
        pace.token_logprob(b, hidden, w, y, loss=la if call == "logprob_with_loss" else None,
                           status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == pace.ERR_INVALID_ARG


@pytest.mark.parametrize("agg", [pace.AGG_TOKEN_MEAN, pace.AGG_SEQ_MEAN_TOKEN_MEAN])
def test_workspace_of_a_larger_batch_serves_a_smaller_one(agg):
    """933,888 rows are one tile a warp of a full launch, 1,200,000 two (in half the blocks)."""
    most, rows, n_seq = 1_200_000, 933_888, 16
    L = pace.lib()
    ws = pace.workspace(L.pace_surrogate_loss_workspace_size(most, n_seq), DEV)
    ws_b = pace.workspace(L.pace_surrogate_backward_workspace_size(most, n_seq), DEV)
    so = np.linspace(0, rows, n_seq + 1).astype(np.int64)
    b = pace.make_batch(to_dev(so), rows)
    lp = torch.zeros(rows, device=DEV)
    reward = (np.arange(n_seq) % 2).astype(np.float32)
    loss = torch.zeros(1, dtype=torch.float64, device=DEV)
    la = pace.make_loss_args(torch.zeros(rows, device=DEV), to_dev(reward), n_seq,
                             pace.loss_params(agg=agg), loss)
    status = pace.new_status(DEV)
    pace.surrogate_loss(b, lp, la, ws=ws, status=status)
    pace.surrogate_backward(b, lp, la, ws=ws_b, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0


def _layout(kind, rng):
    if kind == "short":      # more sequences than a walker holds, in every tile, and empty ones
        return rng.integers(0, 6, size=1200)
    if kind == "edges":      # tile edges on sequence edges, empties there too
        return np.array([256, 0, 0, 255, 1, 0, 512, 257, 0, 511, 1, 1, 0, 2, 254, 0])
    if kind == "one":
        return np.array([1])
    if kind == "gap":        # long sequences between short ones
        return np.array([0, 3000, 1, 5000, 0, 1, 2, 4097, 31, 0])
    if kind == "empties":    # runs of empty sequences around the 31 that a walker holds
        runs = [np.zeros(k, np.int64) for k in (40, 30, 31, 32, 61, 62, 63, 93, 3000, 125)]
        full = [3, 253, 1, 300, 7, 2000, 1, 200, 12]
        return np.concatenate([x for r, f in zip(runs, full) for x in (r, [f])] + runs[-1:])
    return rng.integers(0, 4000, size=608)  # several tiles a warp


@pytest.mark.parametrize("kind,G", [("short", 40), ("short", 5), ("edges", 8), ("one", 1),
                                    ("gap", 2), ("long", 32), ("long", 1)])
@pytest.mark.parametrize("agg", [pace.AGG_TOKEN_MEAN, pace.AGG_SEQ_MEAN_TOKEN_MEAN])
@pytest.mark.parametrize("masked", [False, True])
def test_row_tiles_of_any_layout(kind, G, agg, masked):
    """The loss, the ratios and the derivative over sequences of every length relative to
    the 256-row tiles.  Ratios lie off the clip edges, so fp32 and fp64 take the same
    branch; a term is within 16 roundings of fp32 (expf 2 ulp), sums are fp64."""
    rng = np.random.default_rng(G)
    lens = _layout(kind, rng)
    so = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    n_seq, n = lens.size, int(so[-1])
    lp = (-3.0 * rng.random(n)).astype(np.float32)
    d = rng.choice([-25.0, -0.5, -0.1, 0.0, 0.1, 0.2, 0.4, 2.0, 3.0], size=n)
    behav = (lp - d).astype(np.float32)
    mask = (rng.random(n) < 0.6).astype(np.uint8) if masked else None
    acc = (rng.random(n_seq) < 0.7).astype(np.uint8) if masked else None
    reward = rng.choice([0.0, 0.5, 1.0], size=n_seq).astype(np.float32)
    params = pace.loss_params(agg=agg)
    loss = torch.full((1,), 7.0, dtype=torch.float64, device=DEV)
    ratio = torch.full((n,), 7.0, dtype=torch.float32, device=DEV)
    adv = torch.empty(n_seq, dtype=torch.float32, device=DEV)
    la = pace.make_loss_args(to_dev(behav), to_dev(reward), G, params, loss, adv_out=adv,
                             ratio_out=ratio)
    b = pace.make_batch(to_dev(so), n, seq_accepted=None if acc is None else to_dev(acc),
                        mask=None if mask is None else to_dev(mask))
    status = pace.new_status(DEV)
    dlp = torch.full((n,), 7.0, dtype=torch.float32, device=DEV)
    pace.surrogate_loss(b, to_dev(lp), la, status=status)
    pace.surrogate_backward(b, to_dev(lp), la, dlp=dlp, status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    _, oadv = oracle.group_advantages(reward, G, seq_accepted=acc, eps=float(np.float32(1e-6)))
    np.testing.assert_array_equal(as_np(adv), oadv.astype(np.float32))
    # the oracle takes the rounded differences the kernel sees
    kw = dict(mask=mask, seq_accepted=acc, eps_low=float(np.float32(0.2)),
              eps_high=float(np.float32(0.28)), agg=agg)
    a32 = oadv.astype(np.float32)
    d32 = (lp - behav).astype(np.float64)
    st, oloss, oratio, oterm = oracle.surrogate(d32, np.zeros(n), so, a32, **kw)
    assert st == 0
    st, odlp = oracle.surrogate_grad(d32, np.zeros(n), so, a32, **kw)
    assert st == 0
    unit = 16 * 2.0 ** -24
    assert abs(float(loss.item()) - oloss) <= unit * max(np.abs(oterm).max(initial=0.0), 1e-30)
    assert (np.abs(as_np(ratio) - oratio) <= unit * oratio).all()
    assert (np.abs(as_np(dlp) - odlp) <= unit * np.abs(odlp)).all()


@pytest.mark.parametrize("agg", [pace.AGG_TOKEN_MEAN, pace.AGG_SEQ_MEAN_TOKEN_MEAN])
@pytest.mark.parametrize("masked", [False, True])
def test_runs_of_empty_sequences(agg, masked):
    assert _layout("empties", None).size == 3546
    test_row_tiles_of_any_layout("empties", 9, agg, masked)


@pytest.mark.parametrize("call", ["loss", "derivative", "list"])
def test_runs_of_empty_sequences_are_not_walked(call):
    """200,000 empty sequences between two of 5,000 rows: walked one by one they took 23 ms
    in the loss's launch and 42 in the derivative's two."""
    n, E = 10_000, 200_000
    so = np.full(E + 3, 5000, np.int64)
    so[0], so[-1] = 0, n
    b = pace.make_batch(to_dev(so), n)
    lp = torch.zeros(n, device=DEV)
    loss = torch.zeros(1, dtype=torch.float64, device=DEV)
    la = pace.make_loss_args(lp, torch.ones(E + 2, device=DEV), 2, pace.loss_params(), loss)
    acc = torch.ones(E + 2, dtype=torch.uint8, device=DEV)
    hidden = torch.zeros((n, 64), dtype=torch.bfloat16, device=DEV)
    w, y = hidden[:64], torch.zeros(n, dtype=torch.int32, device=DEV)
    masked = pace.make_batch(to_dev(so), n, seq_accepted=acc)
    run = {"loss": lambda: pace.surrogate_loss(b, lp, la),
           "derivative": lambda: pace.surrogate_backward(b, lp, la),
           "list": lambda: pace.token_logprob(masked, hidden, w, y)}[call]
    times = []
    for _ in range(8):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        run()
        e1.record()
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1))
    assert min(times) < 3.0  # ms


def test_short_sequences_share_a_tile():
    """The sequence mean over 5,000 rows of 1,000 sequences: with a tile's pieces taken one
    by one the loss took 75 us and the derivative 95, shared out among the lanes 20 and 17."""
    n, n_seq = 5000, 1000
    so = to_dev(np.arange(n_seq + 1, dtype=np.int64) * (n // n_seq))
    b = pace.make_batch(so, n)
    lp, dlp = torch.zeros(n, device=DEV), torch.empty(n, device=DEV)
    loss = torch.zeros(1, dtype=torch.float64, device=DEV)
    la = pace.make_loss_args(lp, torch.rand(n_seq, device=DEV), 8,
                             pace.loss_params(agg=pace.AGG_SEQ_MEAN_TOKEN_MEAN), loss)
    L = pace.lib()
    ws = pace.workspace(L.pace_surrogate_loss_workspace_size(n, n_seq), DEV)
    ws_b = pace.workspace(L.pace_surrogate_backward_workspace_size(n, n_seq), DEV)
    pace.surrogate_loss(b, lp, la, ws=ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(10):
            pace.surrogate_loss(b, lp, la, ws=ws)
            pace.surrogate_backward(b, lp, la, dlp=dlp, ws=ws_b)
    times = []
    for _ in range(8):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        graph.replay()
        e1.record()
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1) / 10)
    assert min(times) < 0.09  # ms


@pytest.mark.parametrize("agg", [pace.AGG_TOKEN_MEAN, pace.AGG_SEQ_MEAN_TOKEN_MEAN])
@pytest.mark.parametrize("n", [8 * 256, 10_000])
def test_rows_at_any_alignment(agg, n):
    """Arrays that begin off the 32-byte (masks: 8-byte) boundary are read row by row;
    every output has the same bits as from aligned ones, and rows around are not touched."""
    rng = np.random.default_rng(n)
    lens = rng.multinomial(n, np.ones(16) / 16)
    so = to_dev(np.concatenate([[0], np.cumsum(lens)]).astype(np.int64))
    lp, behav = (torch.from_numpy(rng.standard_normal(n).astype(np.float32)) for _ in range(2))
    mask = torch.from_numpy((rng.random(n) < 0.7).astype(np.uint8))
    reward = to_dev(rng.random(16).astype(np.float32))

    def run(shift):
        def at(x):
            y = torch.full((n + 16,), 9, dtype=x.dtype, device=DEV)
            y[shift:shift + n] = x.to(DEV)
            return y[shift:shift + n]
        loss = torch.zeros(1, dtype=torch.float64, device=DEV)
        ratio, dlp = (torch.full((n + 16,), 5.0, dtype=torch.float32, device=DEV)
                      for _ in range(2))
        la = pace.make_loss_args(at(behav), reward, 8, pace.loss_params(agg=agg), loss,
                                 ratio_out=ratio[shift:shift + n])
        b = pace.make_batch(so, n, mask=at(mask))
        x = at(lp)
        pace.surrogate_loss(b, x, la)
        pace.surrogate_backward(b, x, la, dlp=dlp[shift:shift + n])
        torch.cuda.synchronize()
        for y in (ratio, dlp):
            assert (y[:shift] == 5.0).all() and (y[shift + n:] == 5.0).all()
        return loss, ratio[shift:shift + n], dlp[shift:shift + n]

    want = run(0)
    for shift in (1, 2, 4, 7, 8):
        for a, b in zip(run(shift), want):
            assert torch.equal(a, b), shift
