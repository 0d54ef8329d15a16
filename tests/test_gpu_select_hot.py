"""Counting, choosing and managing hot keys at the sizes where the parts hand over: the block's own table of keys, bins of
counts that are cut finer, ties on the lowest chosen count, stretches of keys, and lists around the one-block limit."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import REPLICATE, SINGLE, Oracle
from paper_2104_00501_b200 import binding
from tests.common import dev_keys, host_keys

pytestmark = pytest.mark.gpu


def _top(counts, k):
    return np.lexsort((np.arange(len(counts)), -counts))[:k].astype(np.uint32)


def _check(s, counts, tops, factors=()):
    assert np.array_equal(s.counts().cpu().numpy(), counts)
    for k in tops:
        assert np.array_equal(host_keys(s.select_hot(True, k)), _top(counts, k)), k
    for f in factors:
        m = int((counts * len(counts) > f * counts.sum()).sum())       # far below 2^63
        assert np.array_equal(host_keys(s.select_hot(False, f)), _top(counts, m)), f


@pytest.mark.parametrize("nk", [1, 2, 2047, 2049, 300_001])
def test_counts_and_choices_of_every_size(nk):
    rng = np.random.default_rng(nk)
    s = binding.Store(nk, 4, sync_interval=0)
    counts = np.zeros(nk, np.int64)
    _check(s, counts, [1, nk // 2, nk, nk + 7], [0, 1])               # nothing counted yet: all keys tie
    for n in (1, 1023, 4097, 700_003):
        keys = np.where(rng.random(n) < 0.5, rng.zipf(1.3, n) % nk, rng.integers(0, nk, n)).astype(np.uint32)
        s.count_accesses(dev_keys(keys))
        counts += np.bincount(keys, minlength=nk)
        if n in (1, 700_003):
            _check(s, counts, sorted({1, 2, 10, nk // 3, nk - 1, nk} - {0}), [1, 2, 3, 100])
    bad = np.array([nk, 0xFFFFFFFF, 0, nk - 1], np.uint32)
    s.count_accesses(dev_keys(bad))
    counts[0] += 1
    counts[nk - 1] += 1
    _check(s, counts, [1, min(nk, 5)])
    assert s.status_check() == -4
    s.close()


@pytest.mark.parametrize("calls", [4, 66])
def test_a_bin_that_holds_too_many_keys_is_cut_finer(calls):
    # 70,000 keys whose counts share one bin: 10 * calls (+ up to 6) accesses each; 33,000 are cut twice
    nk, busy = 100_000, 70_000
    rng = np.random.default_rng(calls)
    s = binding.Store(nk, 4, sync_interval=0)
    named = rng.permutation(nk)[:busy].astype(np.uint32)
    per_call = 10 if calls == 4 else 500
    keys = dev_keys(np.tile(named, per_call))
    for _ in range(calls):
        s.count_accesses(keys)
    counts = np.zeros(nk, np.int64)
    counts[named] = per_call * calls
    more = np.repeat(named, np.arange(busy) % 7)
    s.count_accesses(dev_keys(more))
    counts += np.bincount(more, minlength=nk)
    _check(s, counts, [1, 9_999, 10_001, 40_000, 69_999, 70_001, nk], [1, 2])
    s.close()


@pytest.mark.parametrize("n", [1, 1024, 1025, 4097, 16_384, 16_385, 1_048_577])
def test_lists_around_the_one_block_limit(n):
    nk, L = 60_000, 4
    rng = np.random.default_rng(n)
    o, s = Oracle(nk, L, workers=3), binding.Store(nk, L, workers=3)
    for round_ in range(3):
        up = rng.integers(0, nk, n).astype(np.uint32)                 # repeats included
        down = np.concatenate([up[rng.random(n) < 0.4], rng.integers(0, nk, 50).astype(np.uint32)])
        for keys, technique in ((up, (REPLICATE, binding.REPLICATE)), (down, (SINGLE, binding.SINGLE))):
            o.set_management(keys, technique[0])
            s.set_management(dev_keys(keys), technique[1])
            assert np.array_equal(host_keys(s.hot_keys()), o.hot_keys())
    s.close()


def test_setting_the_management_leaves_the_stream_idle():
    # whatever way the call returns: nothing replicated, an empty list, a refused list, the ordinary ways
    nk = 100_000
    s = binding.Store(nk, 8, workers=4, max_device_mib=12)
    few, many = dev_keys(np.arange(64)), dev_keys(np.arange(80_000))
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def idle_after(keys, technique, refused=False):
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)                          # about 50 ms that the call has to wait for
            if refused:
                with pytest.raises(binding.NupsError) as e:
                    s.set_management(keys, technique)
                assert e.value.code == binding.ENOMEM
            else:
                s.set_management(keys, technique)
            return stream.query()

    assert idle_after(few, binding.SINGLE)                          # no key is replicated
    assert idle_after(few[:0], binding.REPLICATE)
    assert idle_after(many, binding.REPLICATE, refused=True)        # 13 MB of replicas
    assert idle_after(few, binding.REPLICATE)
    assert idle_after(many, binding.REPLICATE, refused=True)
    assert idle_after(few[:10].contiguous(), binding.SINGLE)
    assert s.stats()["hot_slots"] == 54
    stream.synchronize()
    s.close()


def test_results_are_copied_where_no_kernel_should_write():
    # page-locked host memory stands for all memory that is not the store's GPU's: no kernel writes the counts to it
    nk = 5001
    rng = np.random.default_rng(1)
    s = binding.Store(nk, 4, sync_interval=0)
    keys = (rng.zipf(1.3, 20_000) % nk).astype(np.uint32)
    s.count_accesses(dev_keys(keys))
    counts = np.bincount(keys, minlength=nk)
    lib, h, stream = binding.load(), s._s, torch.cuda.current_stream()
    out = torch.zeros(nk, dtype=torch.int64).pin_memory()
    before = s.stats()["launches"]
    assert lib.nups_get_counts(h, out.data_ptr(), stream.cuda_stream) == binding.OK
    assert s.stats()["launches"] == before
    stream.synchronize()
    assert np.array_equal(out.numpy(), counts)
    for off in (0, 1):                                               # the GPU's own memory, also where 16-byte stores do not fit
        buf = torch.zeros(nk + 1, dtype=torch.int64, device="cuda")
        assert lib.nups_get_counts(h, buf[off:].data_ptr(), stream.cuda_stream) == binding.OK
        assert np.array_equal(buf[off:off + nk].cpu().numpy(), counts)
    hot, n = torch.zeros(nk, dtype=torch.int32).pin_memory(), C.c_uint64()
    for by_topk, param, want in ((1, 100, 100), (0, 1, int((counts * nk > counts.sum()).sum()))):
        assert lib.nups_select_hot(h, by_topk, param, hot.data_ptr(), C.byref(n), stream.cuda_stream) == binding.OK
        assert n.value == want
        assert np.array_equal(hot.numpy()[:want].view(np.uint32), _top(counts, want))
    assert s.status_check() == 0
    s.close()
