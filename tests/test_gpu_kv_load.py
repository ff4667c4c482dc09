"""kv_state_load through its staging buffer is bit-exact: empty, one entry, and
one entry beyond what is staged at a time (32 MiB: 65536 entries of this
shape), into the second row and last layer, with the neighbours untouched."""
import numpy as np
import pytest

import synth
from gpu_engine import GpuEngine, GpuShard

pytestmark = pytest.mark.gpu


def test_load_is_bit_exact_across_stages():
    shape = synth.TINY
    g = GpuShard(shape, synth.make_weights(shape, 3))
    eng = GpuEngine(g, 2, 65600)
    rng = np.random.default_rng(4)
    mark = rng.integers(0, 1 << 16, (7, 2, 64), dtype=np.uint16)
    eng.load(0, 1, mark, mark + 1)
    eng.load(1, 0, mark + 2, mark + 3)
    for n in (0, 1, 65537):
        k = rng.integers(0, 1 << 16, (n, 2, 64), dtype=np.uint16)
        v = rng.integers(0, 1 << 16, (n, 2, 64), dtype=np.uint16)
        eng.load(1, 1, k, v)
        assert eng.length(1) == n
        rk, rv = eng.read(1, 1, 0, n)
        assert np.array_equal(rk, k) and np.array_equal(rv, v)
    rk, rv = eng.read(0, 1, 0, 7)
    assert np.array_equal(rk, mark) and np.array_equal(rv, mark + 1)
    rk, rv = eng.read(1, 0, 0, 7)
    assert np.array_equal(rk, mark + 2) and np.array_equal(rv, mark + 3)
    eng.close()
    g.close()
