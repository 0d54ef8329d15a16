"""The ordered push at the sizes where its parts hand over to one another: the launch without a sort up to 3,072 rows, tiles
and rounds of the sort, windows of 8, 16 or 32 sorted rows, destinations with more than 32 rows, and their ring of 6 stages."""
import numpy as np
import pytest
import torch

from oracle import REPLICATE, Oracle
from paper_2104_00501_b200 import binding
from tests.common import dev_f32, dev_keys, make_pair, tables_equal

pytestmark = pytest.mark.gpu


def _stream(kind, n, nk, rng):
    if kind == "skewed":
        return (rng.zipf(1.15, n) % nk).astype(np.uint32)
    if kind == "one":
        return np.full(n, nk - 1, np.uint32)
    if kind == "runs":                                     # destinations of 31, 32, 33 and 64, 65 rows, interleaved
        return rng.permutation(np.repeat(np.arange(n // 32 + 1) % nk, np.resize([31, 32, 33, 64, 65], n // 32 + 1))[:n]).astype(np.uint32)
    keys = rng.integers(0, nk, n).astype(np.uint32)        # mostly single rows, some keys out of range
    keys[rng.random(n) < 0.03] = nk + 5
    return keys


@pytest.mark.parametrize("hot_n", [0, 90])
@pytest.mark.parametrize("kind", ["skewed", "one", "runs", "bad"])
@pytest.mark.parametrize("n,L", [(1, 4), (33, 36), (3071, 64), (3072, 132), (3073, 4), (4097, 64), (8193, 32), (20_481, 260), (40_000, 100)])
def test_every_size_matches_the_oracle_bit_for_bit(n, L, kind, hot_n):
    nk, R = 5000, 5
    rng = np.random.default_rng(n + L)
    init = rng.normal(size=(nk, L)).astype(np.float32)
    o, s = make_pair(nk, L, R=R, init=init, deterministic=True)
    if hot_n:
        hot = np.concatenate([np.arange(60), [nk - 1], np.arange(3000, 3000 + hot_n - 61)]).astype(np.uint32)
        o.set_management(hot, REPLICATE)
        s.set_management(dev_keys(hot), binding.REPLICATE)
    keys = _stream(kind, n, nk, rng)
    delta = rng.normal(size=(n, L)).astype(np.float32)
    for _ in range(2):
        o.push(keys, delta)
        s.push(dev_keys(keys), dev_f32(delta))
        o.sync()
        s.sync()
        tables_equal(o, s)
    assert s.status_check() == (-4 if kind == "bad" and n > 1 else 0)


@pytest.mark.parametrize("n", [700, 9001])
@pytest.mark.parametrize("value_bytes,L", [(4, 100), (8, 34), (8, 12)])
def test_two_tables_and_8_byte_values(n, value_bytes, L):
    nk, R = 3000, 3
    rng = np.random.default_rng(n)
    real = np.float64 if value_bytes == 8 else np.float32
    o = Oracle(nk, L, workers=R, with_adagrad=True, value_bytes=value_bytes)
    s = binding.Store(nk, L, workers=R, with_adagrad=True, deterministic=True, value_bytes=value_bytes)
    for which in (0, 1):
        init = rng.normal(size=(nk, L)).astype(real)
        o.table(which)[:] = init
        s.write_table(which, init)
    hot = np.arange(40, dtype=np.uint32)
    o.set_management(hot, REPLICATE)
    s.set_management(dev_keys(hot), binding.REPLICATE)
    keys = (rng.zipf(1.3, n) % nk).astype(np.uint32)
    dv, da = rng.normal(size=(n, L)).astype(real), rng.random((n, L)).astype(real)
    o.push(keys, dv, da)
    s.push(dev_keys(keys), torch.from_numpy(dv).cuda(), torch.from_numpy(da).cuda())
    o.sync()
    s.sync()
    tables_equal(o, s, 0)
    tables_equal(o, s, 1)


def test_more_rows_than_the_tiles_hold_in_one_round():
    # 148 tiles of 2,048 rows are one round; more rows make tiles of several rounds
    nk, L, n = 300_000, 4, 620_001
    rng = np.random.default_rng(3)
    o, s = make_pair(nk, L, R=4, init=rng.normal(size=(nk, L)).astype(np.float32), deterministic=True)
    hot = np.arange(500, dtype=np.uint32)
    o.set_management(hot, REPLICATE)
    s.set_management(dev_keys(hot), binding.REPLICATE)
    keys = (rng.zipf(1.1, n) % nk).astype(np.uint32)
    delta = rng.normal(size=(n, L)).astype(np.float32)
    o.push(keys, delta)
    s.push(dev_keys(keys), dev_f32(delta))
    o.sync()
    s.sync()
    tables_equal(o, s)


@pytest.mark.parametrize("n", [1000, 20_000])
def test_more_destinations_than_32_bits_number(n):
    # the largest store: keys, replicas and the mark of a bad key need more than 32 bits, also for few rows
    nk, L = 0xFFFFFFFF, 4
    if torch.cuda.mem_get_info()[0] < 125 << 30:
        pytest.skip("the store takes 121 GB")
    rng = np.random.default_rng(5)
    s = binding.Store(nk, L, workers=2, deterministic=True)
    named = np.concatenate([np.arange(50), nk - 1 - np.arange(50)]).astype(np.uint32)
    s.set_management(dev_keys(named[::7].copy()), binding.REPLICATE)
    keys = named[rng.integers(0, 100, n)]
    keys[::100] = nk                                       # out of range
    delta = rng.normal(size=(n, L)).astype(np.float32)
    s.push(dev_keys(keys), dev_f32(delta))
    s.sync()
    got = s.pull(dev_keys(named)).cpu().numpy()
    for k, row in zip(named, got):
        # a key's rows in order; replicated keys: each of the two workers' halves in order, then their sum
        cut = (n + 1) // 2
        halves = []
        for rows in (delta[:cut][keys[:cut] == k], delta[cut:][keys[cut:] == k]) if k in named[::7] else (delta[keys == k],):
            acc = np.zeros(L, np.float32)
            for r in rows:
                acc = acc + r
            halves.append(acc)
        assert np.array_equal(row, halves[0] if len(halves) == 1 else halves[0] + halves[1]), k
    assert s.status_check() == -4
    s.close()


@pytest.mark.parametrize("kind", ["skewed", "one", "bad"])
@pytest.mark.parametrize("n,L", [(127, 36), (128, 4), (129, 64), (641, 8)])
def test_small_pushes_at_whole_steps_of_the_scans(n, L, kind):
    test_every_size_matches_the_oracle_bit_for_bit(n, L, kind, 90)


@pytest.mark.parametrize("n", [1, 700, 3072, 9001])
@pytest.mark.parametrize("value_bytes,L", [(4, 100), (8, 34)])
def test_accumulators_alone(n, value_bytes, L):
    # the value delta may be left out: the value table stays as it is
    nk, R = 3000, 3
    rng = np.random.default_rng(n)
    real = np.float64 if value_bytes == 8 else np.float32
    o = Oracle(nk, L, workers=R, with_adagrad=True, value_bytes=value_bytes)
    s = binding.Store(nk, L, workers=R, with_adagrad=True, deterministic=True, value_bytes=value_bytes)
    for which in (0, 1):
        init = rng.normal(size=(nk, L)).astype(real)
        o.table(which)[:] = init
        s.write_table(which, init)
    hot = np.arange(40, dtype=np.uint32)
    o.set_management(hot, REPLICATE)
    s.set_management(dev_keys(hot), binding.REPLICATE)
    keys = (rng.zipf(1.3, n) % nk).astype(np.uint32)
    da = rng.random((n, L)).astype(real)
    o.push(keys, np.zeros((n, L), real), da)
    s.push(dev_keys(keys), None, torch.from_numpy(da).cuda())
    o.sync()
    s.sync()
    tables_equal(o, s, 0)
    tables_equal(o, s, 1)
    assert s.status_check() == 0
