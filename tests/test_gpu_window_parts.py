"""Pulls and fast-mode pushes at the numbers of rows where the warps that share a window of 32 rows change (8, 4, 2, 1), with
repeated keys inside a window, replicated keys, two tables and 8-byte values."""
import numpy as np
import pytest
import torch

from oracle import REPLICATE, Oracle
from paper_2104_00501_b200 import binding
from tests.common import dev_keys

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hot_n", [0, 60])
@pytest.mark.parametrize("value_bytes,L", [(4, 64), (4, 36), (8, 12), (8, 100), (8, 34)])
def test_every_row_is_pulled_and_pushed_once(value_bytes, L, hot_n):
    nk, R = 4000, 5
    rng = np.random.default_rng(L + hot_n)
    real = np.float64 if value_bytes == 8 else np.float32
    o = Oracle(nk, L, workers=R, with_adagrad=True, value_bytes=value_bytes)
    s = binding.Store(nk, L, workers=R, with_adagrad=True, deterministic=False, value_bytes=value_bytes, sync_interval=0)
    for which in (0, 1):
        # multiples of 1/16 up to 2^12: every sum is exact, whatever its order
        init = (rng.integers(-32, 33, size=(nk, L)) / 16).astype(real)
        o.table(which)[:] = init
        s.write_table(which, init)
    if hot_n:
        hot = rng.permutation(nk)[:hot_n].astype(np.uint32)
        o.set_management(hot, REPLICATE)
        s.set_management(dev_keys(hot), binding.REPLICATE)
    # 148 multiprocessors hold 4,736 (two tables: 3,552) warps: windows of 32 rows are shared by 8 up to 18,944 rows, ...
    for n in (1, 31, 33, 257, 14_208, 14_209, 18_944, 18_945, 37_889, 75_777):
        keys = np.where(rng.random(n) < 0.4, rng.zipf(1.3, n) % nk, rng.integers(0, nk, n)).astype(np.uint32)
        keys[n // 2] = nk + 1                                       # out of range
        dv, da = ((rng.integers(-4, 5, size=(n, L)) / 16).astype(real) for _ in range(2))
        two = bool(rng.integers(0, 2))
        o.push(keys, dv, da if two else None)
        s.push(dev_keys(keys), torch.from_numpy(dv).cuda(), torch.from_numpy(da).cuda() if two else None)
        ov, oa = o.pull(keys, with_acc=True)
        gv, ga = s.pull(dev_keys(keys), with_acc=True)
        assert np.array_equal(gv.cpu().numpy(), ov) and np.array_equal(ga.cpu().numpy(), oa), n
        assert np.array_equal(s.pull(dev_keys(keys)).cpu().numpy(), ov), n
        assert s.status_check() == -4
    o.sync()
    s.sync()
    for which in (0, 1):
        assert np.array_equal(s.read_table(which).cpu().numpy(), o.table(which))
    s.close()


@pytest.mark.parametrize("hot_n", [0, 60])
@pytest.mark.parametrize("L", [30, 32, 66, 128])
def test_8_byte_rows_of_a_whole_turn_and_a_little_less_and_more(L, hot_n):
    # a turn takes 128 values of two rows; 64 where rows have at most 32 and no warps share a window
    test_every_row_is_pulled_and_pushed_once(8, L, hot_n)
