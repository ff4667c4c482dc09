"""kv_state_load through its staging buffer is bit-exact: empty, one entry, and
one entry beyond what is staged at a time (32 MiB: 65536 entries of this
shape), into the second row and last layer, with the neighbours untouched; with
little memory for the buffer (pieces with a remainder) and with none."""
import numpy as np
import pytest

import paper_2608_19147_gb300 as pkg
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


ENTRY = 2 * 2 * 2 * 64  # bytes of an entry's K and V


@pytest.mark.parametrize("limit", [0, ENTRY - 1, ENTRY, 3 * ENTRY + 100, 40 * ENTRY])
def test_load_is_bit_exact_with_little_or_no_staging(limit):
    shape = synth.TINY
    w = synth.make_weights(shape, 3)
    g = GpuShard(shape, w)
    eng = GpuEngine(g, 2, 1010)
    pkg.shard_debug_set_load_stage(g.h, limit)
    rng = np.random.default_rng(5)
    mark = rng.integers(0, 1 << 16, (7, 2, 64), dtype=np.uint16)
    eng.load(0, 1, mark, mark + 1)
    for n in (1, 2, 1001, 39):
        k = rng.integers(0, 1 << 16, (n, 2, 64), dtype=np.uint16)
        v = rng.integers(0, 1 << 16, (n, 2, 64), dtype=np.uint16)
        eng.load(1, 1, k, v)
        assert eng.length(1) == n
        rk, rv = eng.read(1, 1, 0, n)
        assert np.array_equal(rk, k) and np.array_equal(rv, v)
    rk, rv = eng.read(0, 1, 0, 7)
    assert np.array_equal(rk, mark) and np.array_equal(rv, mark + 1)
    # the step on host buffers has its staging whatever the loads had
    one = GpuEngine(g, 1, 16)
    out = np.empty((2, shape.hidden), np.uint16)
    h = synth.hidden_in(shape, 1, 0, 2)
    pkg.shard_step_host(g.h, one.st, h, None, [2], np.arange(2, dtype=np.int32), np.ones((1, 2), np.uint8), None, out)
    again = GpuEngine(g, 1, 16)
    assert np.array_equal(out, again.step([2], np.arange(2), np.ones((1, 2), np.uint8), hidden_in=h))
    for e in (one, again, eng):
        e.close()
    g.close()
