"""CUDA path vs oracle: the three workload steps (deterministic mode: values within the stated
tolerance, negatives and access counts bit-exact; fast mode: loss within 1 %)."""
import numpy as np
import pytest
import torch

from oracle import BOUNDED, CONFORM, LONGTERM, REPLICATE
from paper_2104_00501_b200 import inputs
from tests.common import ATOL, RTOL, dev_f32, dev_keys, host_keys, make_pair, tables_close

pytestmark = pytest.mark.gpu


def loss_buf():
    return torch.zeros(1, dtype=torch.float32, device="cuda")


def sgns_data(V, n_tokens, seed):
    c, ctx, counts = inputs.sgns_batch_stream(V, n_tokens, 1.1, seed)
    return inputs.u32(c), inputs.u32(ctx), inputs.integer_weights(counts).numpy().astype(np.uint32)


@pytest.mark.parametrize("L,level,hot_n,interval", [(64, CONFORM, 0, 1), (64, CONFORM, 20, 1), (300, BOUNDED, 20, 3),
                                                    (100, LONGTERM, 10, 2), (8, CONFORM, 5, 1)])
def test_sgns_deterministic_parity(L, level, hot_n, interval):
    V, K, R, batch = 300, 3, 4, 250
    c, ctx, w = sgns_data(V, 400, 0)
    init = inputs.normal_init(2 * V, L, 0.1, 0)
    o, s = make_pair(2 * V, L, R=R, init=init, deterministic=True, sync_interval=interval, count_accesses=True,
                     track_ownership=True)
    if hot_n:
        o.count_accesses(np.concatenate([c, ctx]))
        s.count_accesses(dev_keys(np.concatenate([c, ctx])))
        hot = o.select_hot(True, hot_n)
        assert np.array_equal(host_keys(s.select_hot(True, hot_n)), hot)
        o.set_management(hot, REPLICATE)
        s.set_management(dev_keys(hot), REPLICATE)
    do = o.register_distribution(V, w, V, level, U=4, G=25, seed=3)
    ds = s.register_distribution(V, dev_keys(w), V, level, U=4, G=25, seed=3)
    lb = loss_buf()
    for b in range(0, len(c) - batch, batch):
        lo, negs = o.step_sgns(c[b:b + batch], ctx[b:b + batch], do, K, 0.05, return_negatives=True)
        s.step_sgns(dev_keys(c[b:b + batch]), dev_keys(ctx[b:b + batch]), ds, K, 0.05, lb)
        assert np.array_equal(host_keys(s.last_negatives()), negs)
        assert abs(lb.item() - lo) <= 1e-5 * abs(lo)
    o.sync()
    s.sync()
    tables_close(o, s)
    assert np.array_equal(s.counts().cpu().numpy().astype(np.uint64), o.counts())
    assert s.stats()["steps"] == o.stats()["steps"] and s.stats()["syncs"] == o.stats()["syncs"]
    assert np.abs(o.table() - init).max() > 1e-3


def test_sgns_ragged_and_single_item_batches():
    V, L, K = 50, 12, 2
    c, ctx, w = sgns_data(V, 80, 1)
    init = inputs.normal_init(2 * V, L, 0.2, 1)
    o, s = make_pair(2 * V, L, R=8, init=init, deterministic=True)
    do = o.register_distribution(V, w, V, CONFORM, seed=1)
    ds = s.register_distribution(V, dev_keys(w), V, CONFORM, seed=1)
    lb = loss_buf()
    at = 0
    for n in (1, 3, 33, 129, 7):
        lo = o.step_sgns(c[at:at + n], ctx[at:at + n], do, K, 0.1)
        s.step_sgns(dev_keys(c[at:at + n]), dev_keys(ctx[at:at + n]), ds, K, 0.1, lb)
        assert abs(lb.item() - lo) <= 1e-5 * abs(lo)
        at += n
    tables_close(o, s)


@pytest.mark.parametrize("L,hot_n,K", [(500, 0, 10), (500, 30, 10), (8, 4, 3), (64, 10, 0)])
def test_complex_deterministic_parity(L, hot_n, K):
    E, Rl, R, batch = 400, 12, 4, 100
    h, r, t = [inputs.u32(x) for x in inputs.kge_triples(300, E, Rl, 0.9, 1.2, 0)]
    rng = np.random.default_rng(0)
    init = rng.normal(0, 0.1, size=(E + Rl, L)).astype(np.float32)
    o, s = make_pair(E + Rl, L, R=R, init=init, deterministic=True, with_adagrad=True, count_accesses=True)
    if hot_n:
        hot = np.concatenate([np.arange(E, E + Rl), np.unique(h)[:hot_n]]).astype(np.uint32)
        o.set_management(hot, REPLICATE)
        s.set_management(dev_keys(hot), REPLICATE)
    do = o.register_distribution(0, None, E, CONFORM, seed=9)
    ds = s.register_distribution(0, None, E, CONFORM, seed=9)
    lb = loss_buf()
    for b in range(0, 300, batch):
        sl = slice(b, b + batch)
        lo, negs = o.step_complex(h[sl], r[sl], t[sl], do, K, 0.1, 1e-10, return_negatives=True)
        s.step_complex(dev_keys(h[sl]), dev_keys(r[sl]), dev_keys(t[sl]), ds, K, 0.1, 1e-10, lb)
        assert np.array_equal(host_keys(s.last_negatives()), negs)
        assert abs(lb.item() - lo) <= 1e-5 * abs(lo)
    o.sync()
    s.sync()
    # deterministic mode computes between pull and push in double precision, as the oracle does, so even
    # AdaGrad's first step (which is lr long whatever the gradient's size) agrees: the stated tolerance, every element
    tables_close(o, s, 1)
    tables_close(o, s, 0)
    assert np.abs(o.table(0) - init).max() > 0.05
    assert np.array_equal(s.counts().cpu().numpy().astype(np.uint64), o.counts())


@pytest.mark.parametrize("L,hot_n", [(100, 0), (100, 25), (4, 3)])
def test_mf_deterministic_parity(L, hot_n):
    M, N, R, batch = 500, 200, 4, 512
    i, j, x = inputs.mf_cells(2048, M, N, 0.8, max(L // 4, 2), 0.1, 0)
    i, j, x = inputs.u32(i), inputs.u32(j), x.numpy()
    init = np.random.default_rng(0).normal(0, 0.3, size=(M + N, L)).astype(np.float32)
    o, s = make_pair(M + N, L, R=R, init=init, deterministic=True, count_accesses=True)
    if hot_n:
        o.count_accesses(np.concatenate([i, j]))
        s.count_accesses(dev_keys(np.concatenate([i, j])))
        hot = o.select_hot(True, hot_n)
        o.set_management(hot, REPLICATE)
        s.set_management(dev_keys(hot), REPLICATE)
    lb = loss_buf()
    for b in range(0, 2048, batch):
        sl = slice(b, b + batch)
        lo = o.step_mf(i[sl], j[sl], x[sl], 0.01, 0.01)
        s.step_mf(dev_keys(i[sl]), dev_keys(j[sl]), dev_f32(x[sl]), 0.01, 0.01, lb)
        assert abs(lb.item() - lo) <= 1e-5 * abs(lo)
    o.sync()
    s.sync()
    tables_close(o, s)
    assert np.array_equal(s.counts().cpu().numpy().astype(np.uint64), o.counts())


@pytest.mark.parametrize("L,hot_n,n", [(100, 0, 4096), (100, 25, 4096), (8, 10, 3001), (300, 25, 1500), (300, 25, 6000)])
def test_mf_fast_mode_on_cells_in_column_order(L, hot_n, n):
    # cells visited column by column (Section 5.1): fast mode sums a column's updates over a stretch of cells before
    # it adds them.  One step from the same start: every row's total update is the oracle's up to the races between
    # cells that share a row (second order in the learning rate, which is small here), so a lost or misdirected
    # sum (a whole stretch of a column) cannot hide in the tolerance
    M, N, R = 500, 200, 4
    i, j, x = inputs.mf_cells(n, M, N, 0.8, max(L // 4, 2), 0.1, 0, by_column_of=20 * n)
    assert len(torch.unique_consecutive(j)) < n // 8               # long runs of one column
    i, j, x = inputs.u32(i), inputs.u32(j), x.numpy()
    init = np.random.default_rng(0).normal(0, 0.3, size=(M + N, L)).astype(np.float32)
    o, s = make_pair(M + N, L, R=R, init=init, deterministic=False)
    if hot_n:
        o.count_accesses(np.concatenate([i, j]))
        hot = o.select_hot(True, hot_n)
        o.set_management(hot, REPLICATE)
        s.set_management(dev_keys(hot), REPLICATE)
    lb = loss_buf()
    # a cell may see updates of cells before it, which the oracle's batch step never shows: for a row that c cells
    # share that changes its update by up to lr * c * |row|^2 (first order), so the learning rate is tiny; the
    # absolute term is the fp32 rounding of the stored rows
    lr = 2e-6
    lo = o.step_mf(i, j, x, lr, 0.01)
    s.step_mf(dev_keys(i), dev_keys(j), dev_f32(x), lr, 0.01, lb, by_column=True)
    assert abs(lb.item() - lo) <= 2e-3 * abs(lo)
    o.sync()
    s.sync()
    d_o = o.table(0).astype(np.float64) - init
    d_s = s.read_table(0).cpu().numpy().astype(np.float64) - init
    norm = np.linalg.norm(d_o, axis=1)
    assert np.all(np.linalg.norm(d_s - d_o, axis=1) <= 0.01 * norm + 2e-6)
    assert norm.max() > 2e-5
    assert s.status_check() == 0


@pytest.mark.parametrize("n", [701, 6007])          # below and above one cell per resident warp: the plain kernel and the one for runs
def test_mf_by_column_takes_any_order_bad_keys_and_single_cells(n):
    # independent cells (hardly any runs), keys out of range in the middle and at the end, access counting and the
    # ownership map on: counts are exact, bad cells are skipped and flagged, every row's update is the oracle's
    M, N, L, R = 60, 40, 100, 3
    i, j, x = inputs.mf_cells(n, M, N, 0.8, 8, 0.1, 1)
    i, j, x = inputs.u32(i), inputs.u32(j), x.numpy()
    init = np.random.default_rng(1).normal(0, 0.3, size=(M + N, L)).astype(np.float32)
    o, s = make_pair(M + N, L, R=R, init=init, deterministic=False, count_accesses=True, track_ownership=True)
    hot = np.array([int(i[0]), int(j[0])], np.uint32)
    o.set_management(hot, REPLICATE)
    s.set_management(dev_keys(hot), REPLICATE)
    lb = loss_buf()
    lr = 2e-6                                  # tiny, see test_mf_fast_mode_on_cells_in_column_order
    lo = o.step_mf(i, j, x, lr, 0.01)
    s.step_mf(dev_keys(i), dev_keys(j), dev_f32(x), lr, 0.01, lb, by_column=True)
    assert abs(lb.item() - lo) <= 2e-3 * abs(lo)
    assert s.status_check() == 0
    one = slice(5, 6)
    lo = o.step_mf(i[one], j[one], x[one], lr, 0.01)
    s.step_mf(dev_keys(i[one]), dev_keys(j[one]), dev_f32(x[one]), lr, 0.01, lb, by_column=True)
    assert abs(lb.item() - lo) <= 1e-4 * abs(lo) + 1e-7
    o.sync()
    s.sync()
    d_o = o.table(0).astype(np.float64) - init
    d_s = s.read_table(0).cpu().numpy().astype(np.float64) - init
    norm = np.linalg.norm(d_o, axis=1)
    assert np.all(np.linalg.norm(d_s - d_o, axis=1) <= 0.01 * norm + 2e-6)
    assert norm.max() > 2e-5
    assert np.array_equal(s.counts().cpu().numpy().astype(np.uint64), o.counts())
    # cells with a key out of range change nothing and raise the flag
    before = s.read_table(0).clone()
    bi, bj = i[:40].copy(), j[:40].copy()
    bi[:] = M + N + 3
    bj[-1] = 0xFFFFFFF0
    s.step_mf(dev_keys(bi), dev_keys(bj), dev_f32(x[:40]), lr, 0.01, lb, by_column=True)
    s.sync()
    assert s.status_check() == -4
    assert torch.equal(s.read_table(0), before)


@pytest.mark.parametrize("n", [2003, 6007])
def test_mf_by_column_sends_each_cells_update_to_its_own_workers_replica(n):
    # no merge after the step: a pull from worker q's part of a call sees the stored row plus q's pending updates
    # only, so the replicas must hold exactly the updates of the cells that belong to each worker
    M, N, L, R = 80, 30, 100, 5
    i, j, x = inputs.mf_cells(n, M, N, 0.8, 8, 0.1, 4, by_column_of=30 * n)
    i, j, x = inputs.u32(i), inputs.u32(j), x.numpy()
    init = np.random.default_rng(4).normal(0, 0.3, size=(M + N, L)).astype(np.float32)
    o, s = make_pair(M + N, L, R=R, init=init, deterministic=False, sync_interval=0)
    o.count_accesses(np.concatenate([i, j]))
    hot = o.select_hot(True, 12)
    o.set_management(hot, REPLICATE)
    s.set_management(dev_keys(hot), REPLICATE)
    lr = 2e-6
    o.step_mf(i, j, x, lr, 0.01)
    s.step_mf(dev_keys(i), dev_keys(j), dev_f32(x), lr, 0.01, loss_buf(), by_column=True)
    keys = np.tile(hot, R).astype(np.uint32)                    # item block q of the pull belongs to worker q
    want = o.pull(keys).astype(np.float64) - init[keys]
    got = s.pull(dev_keys(keys)).cpu().numpy().astype(np.float64) - init[keys]
    norm = np.linalg.norm(want, axis=1)
    assert np.all(np.linalg.norm(got - want, axis=1) <= 0.01 * norm + 2e-6)
    per_worker = norm.reshape(R, len(hot))
    assert (per_worker > 1e-5).sum() >= 2 * R                   # several workers hold updates of several keys ...
    assert np.ptp(per_worker, axis=0).max() > 1e-5              # ... and not the same ones


def test_fast_mode_reaches_the_oracles_loss_within_one_percent():
    # replicated + asynchronous mode: same number of epochs, final loss within 1 % of the oracle's
    V, L, K, R, batch = 500, 32, 3, 8, 256
    c, ctx, w = sgns_data(V, 4000, 2)
    init = inputs.normal_init(2 * V, L, 0.1, 2)
    o, s = make_pair(2 * V, L, R=R, init=init, deterministic=False, sync_interval=4)
    o.count_accesses(np.concatenate([c, ctx]))
    hot = o.select_hot(True, 20)
    o.set_management(hot, REPLICATE)
    s.set_management(dev_keys(hot), REPLICATE)
    do = o.register_distribution(V, w, V, BOUNDED, U=4, G=50, seed=3)
    ds = s.register_distribution(V, dev_keys(w), V, BOUNDED, U=4, G=50, seed=3)
    lb = loss_buf()
    lo_hist, ls_hist = [], []
    nb = (len(c) // batch)
    for epoch in range(2):
        for b in range(nb):
            sl = slice(b * batch, (b + 1) * batch)
            lo_hist.append(o.step_sgns(c[sl], ctx[sl], do, K, 0.01))
            s.step_sgns(dev_keys(c[sl]), dev_keys(ctx[sl]), ds, K, 0.01, lb)
            ls_hist.append(lb.item())
    lo, ls = np.mean(lo_hist[-nb:]), np.mean(ls_hist[-nb:])
    assert abs(ls - lo) <= 0.01 * lo
    assert lo < 0.95 * np.mean(lo_hist[:20])
    assert s.status_check() == 0


def test_tiny_sgns_config_full_epoch():
    # config 0: 10,000-word vocabulary (20,000 keys), dim 64, N(0, 0.01) start values, 256k pairs
    # with Zipf(1.1) words, batch 256, 3 CONFORM negatives from unigram^0.75, lr 0.025, top-100 keys
    # replicated, sync every step, one epoch, seed 0
    V, L, K, R, batch = 10000, 64, 3, 8, 256
    c, ctx, counts = inputs.sgns_batch_stream(V, 25700, 1.1, 0)
    c, ctx = inputs.u32(c)[:256000], inputs.u32(ctx)[:256000]
    w = inputs.integer_weights(counts).numpy().astype(np.uint32)
    init = inputs.normal_init(2 * V, L, 0.01, 0)
    o, s = make_pair(2 * V, L, R=R, init=init, deterministic=True, sync_interval=1, count_accesses=True)
    both = np.concatenate([c, ctx])
    o.count_accesses(both)
    s.count_accesses(dev_keys(both))
    hot = o.select_hot(True, 100)
    assert np.array_equal(host_keys(s.select_hot(True, 100)), hot)
    o.set_management(hot, REPLICATE)
    s.set_management(dev_keys(hot), REPLICATE)
    do = o.register_distribution(V, w, V, CONFORM, seed=0)
    ds = s.register_distribution(V, dev_keys(w), V, CONFORM, seed=0)
    lb = torch.zeros(1000, dtype=torch.float32, device="cuda")
    dc, dx = dev_keys(c), dev_keys(ctx)
    lo = []
    for b in range(1000):
        sl = slice(b * batch, (b + 1) * batch)
        lo.append(o.step_sgns(c[sl], ctx[sl], do, K, 0.025))
        s.step_sgns(dc[sl], dx[sl], ds, K, 0.025, lb[b:b + 1])
    ls = lb.cpu().numpy()
    np.testing.assert_allclose(ls, np.array(lo, np.float32), rtol=1e-5)
    tables_close(o, s)
    assert np.array_equal(s.counts().cpu().numpy().astype(np.uint64), o.counts())
    assert s.status_check() == 0


@pytest.mark.parametrize("level", [CONFORM, BOUNDED])
def test_sample_ahead_keeps_the_sample_sequences(level):
    # in fast mode the negatives of several steps are drawn in one launch; whatever else touches the
    # distribution in between (PrepareSample, a step of another size), the keys stay those of the oracle
    V, L, K, R = 400, 16, 3, 4
    c, ctx, w = sgns_data(V, 700, 5)
    init = inputs.normal_init(2 * V, L, 0.1, 5)
    o, s = make_pair(2 * V, L, R=R, init=init, deterministic=False, sync_interval=2)
    do = o.register_distribution(V, w, V, level, U=3, G=20, seed=4)
    ds = s.register_distribution(V, dev_keys(w), V, level, U=3, G=20, seed=4)
    lb = loss_buf()
    at = 0
    plan = [64] * 20 + ["pull"] + [64] * 3 + [100] * 2 + [64] * 18 + ["pull", "pull"] + [33] * 20
    for what in plan:
        if what == "pull":
            ko = o.pull_sample(o.prepare_sample(do, 77), 77, values=False)
            ks = s.pull_sample(s.prepare_sample(ds, 77), 77, values=False)
            assert np.array_equal(host_keys(ks), ko)
            continue
        n = what
        _, negs = o.step_sgns(c[at:at + n], ctx[at:at + n], do, K, 0.01, return_negatives=True)
        s.step_sgns(dev_keys(c[at:at + n]), dev_keys(ctx[at:at + n]), ds, K, 0.01, lb)
        assert np.array_equal(host_keys(s.last_negatives()), negs)
        at += n
    assert s.status_check() == 0


def test_run_sgns_matches_step_by_step():
    # deterministic mode: nups_run_sgns is the step loop, exactly; fast mode: steps between two merges share a
    # launch, negatives and merge cadence stay the same and the loss tracks the oracle's within 1 %
    V, L, K, R, B = 600, 32, 3, 4, 128
    c, ctx, w = sgns_data(V, 2000, 7)
    steps = 40
    c, ctx = c[:steps * B], ctx[:steps * B]
    init = inputs.normal_init(2 * V, L, 0.1, 7)
    o, s = make_pair(2 * V, L, R=R, init=init, deterministic=True, sync_interval=3)
    do = o.register_distribution(V, w, V, BOUNDED, U=4, G=30, seed=2)
    ds = s.register_distribution(V, dev_keys(w), V, BOUNDED, U=4, G=30, seed=2)
    lo = [o.step_sgns(c[t * B:(t + 1) * B], ctx[t * B:(t + 1) * B], do, K, 0.02) for t in range(steps)]
    lb = torch.zeros(steps, device="cuda")
    s.run_sgns(dev_keys(c), dev_keys(ctx), B, ds, K, 0.02, lb)
    np.testing.assert_allclose(lb.cpu().numpy(), np.array(lo, np.float32), rtol=1e-5)
    o.sync()
    s.sync()
    tables_close(o, s)
    assert s.stats()["steps"] == steps and s.stats()["syncs"] == o.stats()["syncs"]

    _, f = make_pair(2 * V, L, R=R, init=init, deterministic=False, sync_interval=3)
    hot = np.unique(c)[:30].astype(np.uint32)
    f.set_management(dev_keys(hot), REPLICATE)
    df = f.register_distribution(V, dev_keys(w), V, BOUNDED, U=4, G=30, seed=2)
    lf = torch.zeros(steps, device="cuda")
    f.run_sgns(dev_keys(c[:17 * B]), dev_keys(ctx[:17 * B]), B, df, K, 0.02, lf[:17])      # ragged split of the run
    f.run_sgns(dev_keys(c[17 * B:]), dev_keys(ctx[17 * B:]), B, df, K, 0.02, lf[17:])
    lf = lf.cpu().numpy()
    assert np.all(np.isfinite(lf)) and abs(lf[-10:].mean() - np.mean(lo[-10:])) <= 0.01 * np.mean(lo[-10:])
    assert f.stats()["steps"] == steps and f.stats()["syncs"] == steps // 3
    # the negatives handed to the last step of the run are the oracle's
    ko = o.pull_sample(o.prepare_sample(do, 50), 50, values=False)
    kf = f.pull_sample(f.prepare_sample(df, 50), 50, values=False)
    assert np.array_equal(host_keys(kf), ko)
    assert f.status_check() == 0


@pytest.mark.parametrize("K", [3, 5])
def test_sgns_clipping_of_replicated_key_updates_matches_the_oracle(K):
    # a learning rate at which the unclipped run blows up (its loss grows step by step): the clipped run stays
    # put, and the CUDA path follows the oracle through it
    from paper_2104_00501_b200 import binding
    V, L, R, batch = 300, 64, 4, 250
    c, ctx, w = sgns_data(V, 400, 7)
    init = inputs.normal_init(2 * V, L, 0.3, 7)
    tables, losses = {}, {}
    for factor in (0.0, 0.7):
        o, s = make_pair(2 * V, L, R=R, init=init, deterministic=True, sync_interval=2)
        s.close()
        s = binding.Store(2 * V, L, workers=R, sync_interval=2, deterministic=True, clip_factor=factor)
        s.write_table(0, init)
        o.set_clipping(factor)
        o.count_accesses(np.concatenate([c, ctx]))
        hot = o.select_hot(True, 25)
        o.set_management(hot, REPLICATE)
        s.set_management(dev_keys(hot), REPLICATE)
        do = o.register_distribution(V, w, V, BOUNDED, U=4, G=50, seed=3)
        ds = s.register_distribution(V, dev_keys(w), V, BOUNDED, U=4, G=50, seed=3)
        lb = loss_buf()
        for b in range(6):
            sl = slice(b * batch, (b + 1) * batch)
            lo = o.step_sgns(c[sl], ctx[sl], do, K, 0.2)
            if factor:
                s.step_sgns(dev_keys(c[sl]), dev_keys(ctx[sl]), ds, K, 0.2, lb)
                assert abs(lb.item() - lo) <= 1e-5 * abs(lo)
            losses.setdefault(factor, []).append(lo)
        o.sync()
        tables[factor] = o.table().copy()
        if factor:
            s.sync()
            tables_close(o, s)
            (so, co), (ss, cs) = o.clip_stats(), s.clip_stats()
            assert co == cs and co > 0 and ss == pytest.approx(so, rel=1e-5)
            assert s.status_check() == 0
        else:
            assert o.clip_stats() == (0.0, 0)
        s.close()
    assert not np.array_equal(tables[0.0], tables[0.7])               # the bound was tight enough to bite
    assert losses[0.7][-1] < losses[0.0][-1]


def test_mf_clipping_matches_the_oracle_and_fast_mode_counts_the_same_updates():
    from paper_2104_00501_b200 import binding
    M, N, L, R, n = 200, 60, 100, 4, 1500
    rng = np.random.default_rng(8)
    rows = inputs.u32(inputs.zipf_keys(n, M, 0.8, 1, "cpu"))
    cols = (M + inputs.u32(inputs.zipf_keys(n, N, 0.8, 2, "cpu"))).astype(np.uint32)
    x = rng.normal(0, 1, n).astype(np.float32)
    init = rng.normal(0, 0.3, (M + N, L)).astype(np.float32)
    hot = np.unique(np.concatenate([rows[:40], cols[:40]])).astype(np.uint32)
    o, s0 = make_pair(M + N, L, R=R, init=init, deterministic=True)
    s0.close()
    o.set_clipping(0.8)
    o.set_management(hot, REPLICATE)
    stores = {}
    for det, by_column in ((True, False), (False, False), (False, True)):      # ordered, fast, fast by column
        s = binding.Store(M + N, L, workers=R, sync_interval=1, deterministic=det, clip_factor=0.8)
        s.write_table(0, init)
        s.set_management(dev_keys(hot), REPLICATE)
        stores[(det, by_column)] = s
    lb = loss_buf()
    for b in range(3):
        sl = slice(b * 500, (b + 1) * 500)
        order = np.argsort(cols[sl], kind="stable")                          # each step's cells column by column
        r_b, c_b, x_b = rows[sl][order], cols[sl][order], x[sl][order]
        lo = o.step_mf(r_b, c_b, x_b, 0.05, 0.01)
        for (det, by_column), s in stores.items():
            s.step_mf(dev_keys(r_b), dev_keys(c_b), dev_f32(x_b), 0.05, 0.01, lb, by_column=by_column)
            if det:
                assert abs(lb.item() - lo) <= 1e-5 * abs(lo)
            else:
                assert abs(lb.item() - lo) <= 0.1 * abs(lo)
    tables_close(o, stores[(True, False)])
    so, co = o.clip_stats()
    for (det, by_column), s in stores.items():
        ss, cs = s.clip_stats()
        assert cs == co
        assert ss == pytest.approx(so, rel=1e-5 if det else 0.25)
        s.close()


def test_fast_mode_with_clipping_tracks_the_clipped_oracle():
    # replicated + asynchronous mode with clipping on, steps taken 16 at a time (the bound is then fixed per launch):
    # the loss stays within 2 % of the oracle's clipped run and exactly the same updates are counted
    from paper_2104_00501_b200 import binding
    V, L, K, R, batch = 500, 32, 3, 8, 256
    c, ctx, w = sgns_data(V, 4000, 2)
    init = inputs.normal_init(2 * V, L, 0.1, 2)
    o, s0 = make_pair(2 * V, L, R=R, init=init, deterministic=False, sync_interval=4)
    s0.close()
    s = binding.Store(2 * V, L, workers=R, sync_interval=4, deterministic=False, clip_factor=1.5)
    s.write_table(0, init)
    o.set_clipping(1.5)
    o.count_accesses(np.concatenate([c, ctx]))
    hot = o.select_hot(True, 20)
    o.set_management(hot, REPLICATE)
    s.set_management(dev_keys(hot), REPLICATE)
    do = o.register_distribution(V, w, V, BOUNDED, U=4, G=50, seed=3)
    ds = s.register_distribution(V, dev_keys(w), V, BOUNDED, U=4, G=50, seed=3)
    nb = len(c) // batch
    lo = [o.step_sgns(c[b * batch:(b + 1) * batch], ctx[b * batch:(b + 1) * batch], do, K, 0.02) for b in range(nb)]
    ls = torch.zeros(nb, device="cuda")
    s.run_sgns(dev_keys(c[:nb * batch]), dev_keys(ctx[:nb * batch]), batch, ds, K, 0.02, ls)
    ls = ls.cpu().numpy()
    assert abs(ls[-20:].mean() - np.mean(lo[-20:])) <= 0.02 * np.mean(lo[-20:])
    (so, co), (ss, cs) = o.clip_stats(), s.clip_stats()
    assert cs == co and ss == pytest.approx(so, rel=0.1)
    assert s.status_check() == 0
    s.close()


@pytest.mark.parametrize("runs", [False, True])
@pytest.mark.parametrize("n,L", [(2960, 100), (2961, 100), (7003, 200), (24_001, 12), (9001, 512)])
def test_mf_by_column_with_bad_keys_at_the_sizes_where_its_batches_change(n, L, runs):
    # 148 multiprocessors: one cell per resident warp (2,960, the plain kernel), then stretches of 2, 4, 12 (9 rounded to whole
    # batches) and 4 cells; runs of one column and columns that change at every cell; keys out of range inside a batch: those
    # cells change nothing.  Cells race here, so a lost update shows only where it is a good part of its row's; cells that
    # cannot race, and stretches of several windows, are in test_gpu_fast_modes.py
    M, N, R = 3000, 900, 3
    i, j, x = inputs.mf_cells(n, M, N, 0.3, 8, 0.1, 2, by_column_of=20 * n if runs else 0)
    i, j, x = inputs.u32(i), inputs.u32(j), x.numpy()
    bad = np.random.default_rng(n).random(n) < 0.02
    init = np.random.default_rng(3).normal(0, 0.3, size=(M + N, L)).astype(np.float32)
    o, s = make_pair(M + N, L, R=R, init=init, deterministic=False)
    hot = np.unique(np.concatenate([i[:20], j[:20]])).astype(np.uint32)
    o.set_management(hot, REPLICATE)
    s.set_management(dev_keys(hot), REPLICATE)
    lr = 2e-6                                  # tiny, see test_mf_fast_mode_on_cells_in_column_order
    bi = i.copy()
    bi[bad] = M + N + 7
    lb = loss_buf()
    s.step_mf(dev_keys(bi), dev_keys(j), dev_f32(x), lr, 0.01, lb, by_column=True)
    assert s.status_check() == -4
    lo = o.step_mf(bi, j, x, lr, 0.01)
    assert abs(lb.item() - lo) <= 2e-3 * abs(lo)
    o.sync()
    s.sync()
    d_o = o.table(0).astype(np.float64) - init
    d_s = s.read_table(0).cpu().numpy().astype(np.float64) - init
    norm = np.linalg.norm(d_o, axis=1)
    assert np.all(np.linalg.norm(d_s - d_o, axis=1) <= 0.01 * norm + 2e-6 * np.sqrt(L / 100 + 1))   # fp32 rounding of every stored value
    assert norm.max() > 2e-5
