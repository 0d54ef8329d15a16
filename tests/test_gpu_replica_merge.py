"""The replica merge where the number of warps that share a slot changes (1, 2, 4, 8; by the rows' width and the number of slots),
with one and two tables, 4- and 8-byte values, up to the most workers, and replicas of which some were not touched."""
import numpy as np
import pytest
import torch

from oracle import REPLICATE, Oracle
from paper_2104_00501_b200 import binding
from tests.common import dev_keys, tables_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,value_bytes,two,R,hot_n", [
    (1028, 4, False, 40, 60), (1028, 4, True, 3, 1184), (1028, 4, False, 3, 1185), (600, 8, True, 40, 50), (500, 4, True, 5, 2368),
    (500, 4, True, 5, 2369), (260, 4, False, 2, 2368), (260, 4, False, 2, 2369), (128, 4, True, 254, 20), (132, 8, False, 33, 30)])
def test_the_merged_tables_are_the_oracles(L, value_bytes, two, R, hot_n):
    nk = 4000
    rng = np.random.default_rng(L + R)
    real = np.float64 if value_bytes == 8 else np.float32
    o = Oracle(nk, L, workers=R, with_adagrad=two, value_bytes=value_bytes)
    s = binding.Store(nk, L, workers=R, with_adagrad=two, deterministic=True, value_bytes=value_bytes, sync_interval=0)
    for which in range(2 if two else 1):
        init = rng.normal(size=(nk, L)).astype(real)
        o.table(which)[:] = init
        s.write_table(which, init)
    hot = rng.permutation(nk)[:hot_n].astype(np.uint32)
    o.set_management(hot, REPLICATE)
    s.set_management(dev_keys(hot), binding.REPLICATE)
    for n in (3, 7 * hot_n + 1, 500):                      # few, most and some replicas touched
        keys = np.where(rng.random(n) < 0.8, hot[rng.integers(0, hot_n, n)], rng.integers(0, nk, n)).astype(np.uint32)
        dv, da = (rng.normal(size=(n, L)).astype(real) for _ in range(2))
        o.push(keys, dv, da if two else None)
        s.push(dev_keys(keys), torch.from_numpy(dv).cuda(), torch.from_numpy(da).cuda() if two else None)
        for _ in range(2):                                 # a merge of nothing changes nothing
            o.sync()
            s.sync()
        for which in range(2 if two else 1):
            tables_equal(o, s, which)
    assert s.status_check() == 0
    s.close()
