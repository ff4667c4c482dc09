"""GPU parity of the step's attention at the edges of its work split, against
the oracle at the fixed bar: cache lengths around the 16-entry blocks and the
64-entry chunks, query tiles of 8 (one, several, more than one pass of 64),
rows cut into many chunks (merged by one CTA or shared out; one per CTA or in
runs), whole rows as units (more request-head pairs than CTAs, more entries than one staged
window), entries that no query sees for a whole item, and large or tiny
queries (their rows are scaled before they are split)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_engine import GpuEngine, GpuShard, assert_close

pytestmark = pytest.mark.gpu

# heads, kv heads, head dim, new tokens per request, cache entries per request
CASES = {
    "empty": (4, 2, 64, [1], [0]),
    "block-1": (4, 2, 128, [1], [14]),
    "block": (4, 2, 128, [1], [15]),
    "block+1": (4, 2, 64, [1], [16]),
    "item": (4, 4, 128, [1], [63]),
    "item+1": (4, 4, 64, [1], [64]),
    "new-over-items": (8, 2, 128, [9], [60]),
    "tile+1": (9, 1, 64, [1], [33]),
    "five-tiles": (8, 1, 128, [5], [190]),
    "two-passes": (16, 1, 64, [7], [300]),
    "four-passes": (16, 1, 128, [16], [40]),
    "many-items": (8, 8, 64, [1], [5000]),
    "shared-merge": (16, 2, 128, [4], [2999]),
    "whole-rows": (16, 16, 64, [1] * 10, [1100, 1023, 1024, 1, 17, 900, 64, 1090, 300, 0]),
    "uneven": (8, 2, 128, [3, 1, 5, 2], [700, 3, 129, 2049]),
    "two-passes-shared-merge": (16, 1, 64, [9], [2500]),
    "runs": (8, 4, 128, [2, 1, 3, 1], [2100, 1500, 1800, 2600]),
}


def _shape(name, scale=1.0):
    hq, hkv, d, _, _ = CASES[name]
    return synth.ShardShape(name, 1, 256, hq, hkv, d, 320, 64, 0.06 * scale, 0, 1e-5, 10000.0, 8192)


def _run(name, mask_of, w, shape):
    _, _, _, n_new, lens = CASES[name]
    cap = max(l + n for l, n in zip(lens, n_new)) + 3
    g = GpuShard(shape, w)
    eng = GpuEngine(g, len(lens), cap)
    ref = oracle.OracleShard(shape, w).state(len(lens), cap)
    for b, n in enumerate(lens):
        k, v = synth.kv_prefill(shape, 5, b, n, 0)
        eng.load(b, 0, k, v)
        assert ref.load(b, 0, k, v) == 0
    h = synth.hidden_in(shape, 6, 0, sum(n_new))
    pos = np.concatenate([np.arange(l, l + n) for l, n in zip(lens, n_new)]).astype(np.int32)
    mask = np.ones((len(lens), cap), np.uint8)
    for b, (l, n) in enumerate(zip(lens, n_new)):
        mask[b, :l] = mask_of(b, l)
    got = eng.step(n_new, pos, mask, hidden_in=h)
    rc, want, _ = ref.step(n_new, pos, mask, hidden_in=h)
    assert rc == 0
    assert_close(got, want, what=name)
    for b, (l, n) in enumerate(zip(lens, n_new)):  # the appended entries: within one fp16 rounding
        for a, o in zip(eng.read(b, 0, l, n), ref.read(b, 0, l, n)):
            a, o = (x.view(np.float16).astype(np.float64) for x in (a, o))
            assert np.abs(a - o).max() <= 2e-3 * max(1.0, np.abs(o).max()), (name, b)
    eng.close()
    g.close()


@pytest.mark.parametrize("name", CASES)
def test_attention_edges(name):
    rng = np.random.default_rng(1)
    shape = _shape(name)
    _run(name, lambda b, l: rng.random(l) < 0.8, synth.make_weights(shape, 3), shape)


@pytest.mark.parametrize("name", ["item+1", "uneven", "shared-merge", "whole-rows", "two-passes-shared-merge", "runs"])
def test_attention_items_nobody_sees(name):
    """Only the last 10 cached entries are visible: whole items contribute nothing."""
    shape = _shape(name)
    _run(name, lambda b, l: np.arange(l) >= l - 10, synth.make_weights(shape, 3), shape)


@pytest.mark.parametrize("scale", [2.0 ** -12, 8.0])
def test_attention_query_scales(scale):
    """q weights far from the usual size: tiny scores, and scores that single out one entry."""
    shape = _shape("five-tiles")
    w = synth.make_weights(shape, 3)
    q = w.layers[0].matrices[0]
    q.scales[:] = (q.scales.view(np.float16).astype(np.float32) * scale).astype(np.float16).view(np.uint16)
    _run("five-tiles", lambda b, l: np.ones(l), w, shape)


@pytest.mark.parametrize("n_new", [1, 3])
def test_a_key_at_minus_infinity_against_its_queries_has_no_weight(n_new):
    """A cached key that overflowed to an infinity, of the sign that gives its head's queries a score of minus
    infinity: the entry has weight 0, as in the oracle, and the outputs stay finite."""
    shape = synth.ShardShape("inf", 1, 256, 4, 4, 64, 320, 64, 0.06, 0, 1e-5, 10000.0, 8192)
    w = synth.make_weights(shape, 17)
    L, entry, dim = 80, 21, 5
    h16 = synth.hidden_in(shape, 8, 0, 1).repeat(n_new, 0)  # one token's queries at one position: one sign per head
    pos, mask = np.full(n_new, L, np.int32), np.ones((1, L + n_new), np.uint8)
    k, v = synth.kv_prefill(shape, 5, 0, L, 0)

    def outputs(state):
        state.load(0, 0, k, v)
        return state.step([n_new], pos, mask, hidden_in=h16)

    ref = oracle.OracleShard(shape, w)
    for head in range(4):
        for inf in (0x7C00, 0xFC00):
            k[entry, head, dim] = inf
            rc, want, _ = outputs(ref.state(1, L + n_new))
            if rc == 0 and np.isfinite(want.view(np.float16)).all():
                break
        else:
            pytest.fail("no sign of the infinity gives a score of minus infinity")
    g = GpuShard(shape, w)
    got = outputs(GpuEngine(g, 1, L + n_new))
    assert_close(got, want, what="key at minus infinity")
    g.close()
