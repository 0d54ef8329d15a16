"""Pooled reuse at the pool sizes and use frequencies where a pass's 32-step groups, the warps of a block and the pool's draws
end: the sampled keys are the oracle's, whatever stretches of the stream the handles take."""
import numpy as np
import pytest

from oracle import BOUNDED, Oracle
from paper_2104_00501_b200 import binding, inputs
from tests.common import dev_keys, host_keys

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("U", [1, 3, 16, 17, 40])
@pytest.mark.parametrize("G", [1, 2, 31, 32, 33, 64, 65, 250, 511, 513, 1023, 1024])
def test_sampled_keys_are_the_oracles(U, G):
    nk, R = 6000, 3
    w = inputs.zipf_integer_weights(5000, 0.9).numpy().astype(np.uint32)
    o, s = Oracle(nk, 4, workers=R), binding.Store(nk, 4, workers=R, sync_interval=0)
    do = o.register_distribution(700, w, 5000, BOUNDED, U=U, G=G, seed=U * 2000 + G)
    ds = s.register_distribution(700, dev_keys(w), 5000, BOUNDED, U=U, G=G, seed=U * 2000 + G)
    for n in (1, 3 * G + 2, 5, 3 * U * G + 17):
        ho, hs = o.prepare_sample(do, n), s.prepare_sample(ds, n)
        assert np.array_equal(host_keys(s.pull_sample(hs, n, values=False)), o.pull_sample(ho, n, values=False)), n
    s.close()
