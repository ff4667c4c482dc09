"""A request's step gives the same bits alone and among others, for caches that
are cut into several attention chunks: rows whose chunks find a CTA each only
when they are alone, units of several chunks (a query tile of a chunk per warp;
pieces of one block and of several; entries staged in several goes; chunk by
chunk where the queries or a chunk's scores are too many), whole rows as units,
several units per CTA, and rows with masked entries and whole masked chunks."""
import numpy as np
import pytest

import synth
from gpu_engine import GpuEngine, GpuShard

pytestmark = pytest.mark.gpu

# heads, kv heads, head dim, new tokens per request, cache entries per request
CASES = {
    "decode": (32, 8, 128, [1] * 8, [2048, 5, 700, 64, 129, 1500, 333, 1642]),
    "decode-d64": (8, 8, 64, [1] * 5, [1217, 2400, 300, 15, 1023]),
    "verify": (32, 8, 128, [3, 1, 5, 2], [2049, 700, 129, 3000]),
    "eight-queries": (64, 8, 128, [1] * 6, [900, 4096, 2500, 777, 1600, 64]),
    "staged-in-parts": (16, 8, 64, [1] * 16, [1990 + 13 * i for i in range(16)]),
    "many-queries": (16, 1, 64, [6, 1, 3], [5000, 900, 2500]),
    "long-chunks": (8, 8, 128, [1, 2, 1], [9000, 12000, 10000]),
    "whole-rows": (16, 16, 64, [1] * 10, [1100, 1023, 1024, 1, 17, 900, 64, 1090, 300, 0]),
}


@pytest.mark.parametrize("name", list(CASES))
def test_a_row_has_the_same_bits_alone_and_batched(name):
    hq, hkv, d, n_new, lens = CASES[name]
    shape = synth.ShardShape(name, 1, 256, hq, hkv, d, 320, 64, 0.06, 0, 1e-5, 10000.0, 16384)
    sh = GpuShard(shape, synth.make_weights(shape, 21))
    cap = max(l + n for l, n in zip(lens, n_new))
    rng = np.random.default_rng(4)
    hidden = [synth.hidden_in(shape, 30 + b, 0, n) for b, n in enumerate(n_new)]
    kv = [synth.kv_prefill(shape, 9, b, l, 0) for b, l in enumerate(lens)]
    mask = np.zeros((len(lens), cap), np.uint8)
    for b, (l, n) in enumerate(zip(lens, n_new)):
        mask[b, :l + n] = 1
        if b % 3 == 1:
            mask[b, :l] = rng.random(l) < 0.8
        if b % 3 == 2:
            mask[b, :l // 2] = 0
    pos = [np.arange(l, l + n, dtype=np.int32) for l, n in zip(lens, n_new)]
    both = GpuEngine(sh, len(lens), cap)
    for b, (k, v) in enumerate(kv):
        both.load(b, 0, k, v)
    got = both.step(n_new, np.concatenate(pos), mask, hidden_in=np.concatenate(hidden))
    assert np.isfinite(got.view(np.float16).astype(np.float32)).all()
    t = 0
    for b, n in enumerate(n_new):
        alone = GpuEngine(sh, 1, cap)
        alone.load(0, 0, *kv[b])
        want = alone.step([n], pos[b], mask[b], hidden_in=hidden[b])
        assert np.array_equal(want, got[t:t + n]), "row %d of %d entries" % (b, lens[b])
        alone.close()
        t += n
    both.close()
    sh.close()
