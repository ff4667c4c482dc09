"""GPU parity of shard_prefill where its projections change shape, against the
oracle's step of the same tokens at the fixed bar: one token to more than one
chunk, every token tile (32, 64, 128), K in one to four parts, a SwiGLU width
that is no multiple of 32, each quantisation group, one query head per kv head
and sixteen, a prompt behind a cache with masked entries, and buffers that are
aligned to their values only."""
import numpy as np
import pytest
import torch

import oracle
import paper_2608_19147_gb300 as pkg
import synth
from gpu_engine import GpuShard, assert_close, to_dev

pytestmark = pytest.mark.gpu

SHAPES = {
    "g128": synth.ShardShape("g128", 2, 1024, 8, 2, 128, 2104, 128, 0.03, 0, 1e-5, 10000.0, 4096),
    "g64": synth.ShardShape("g64", 1, 520, 16, 1, 64, 333, 64, 0.03, 0, 1e-5, 10000.0, 4096),
    "g32": synth.ShardShape("g32", 1, 2048, 4, 4, 64, 1504, 32, 0.03, 0, 1e-5, 10000.0, 4096),
}


def _run(name, S, P, offset=0):
    shape = SHAPES[name]
    w = synth.make_weights(shape, 31)
    g = GpuShard(shape, w)
    st = pkg.kv_state_alloc(g.h, 2, P + S + 5)
    ref = oracle.OracleShard(shape, w).state(1, P + S + 5)
    for l in range(shape.n_layers):
        k, v = synth.kv_prefill(shape, 7, 0, P, l)
        pkg.kv_state_load(st, 1, l, k, v)
        assert ref.load(0, l, k, v) == 0
    h = synth.hidden_in(shape, 8, 0, S)
    mask = np.ones(P + S, np.uint8)
    mask[:P] = np.random.default_rng(2).random(P) < 0.7
    pos = np.arange(P, P + S, dtype=np.int32)
    d_in = torch.zeros(S * shape.hidden + 8, dtype=torch.int16, device="cuda")
    d_in[offset:offset + h.size] = to_dev(h).reshape(-1)
    d_out = torch.zeros(S * shape.hidden + 8, dtype=torch.int16, device="cuda")
    d_pos, d_mask = to_dev(pos), to_dev(mask)
    s = torch.cuda.current_stream().cuda_stream
    pkg.shard_prefill(g.h, st, 1, d_in.data_ptr() + 2 * offset, None, S, d_pos.data_ptr(), d_mask.data_ptr(), P + S,
                      d_out.data_ptr() + 2 * offset, s)
    pkg.shard_sync_status(g.h, s)
    got = d_out[offset:offset + h.size].cpu().numpy().view(np.uint16).reshape(h.shape)
    # the oracle's step takes any number of tokens of one request
    rc, want, _ = ref.step([S], pos, mask, hidden_in=h)
    assert rc == 0
    assert_close(got, want, what="%s S=%d P=%d" % (name, S, P))
    pkg.kv_state_free(st)
    g.close()


@pytest.mark.parametrize("S,P", [(1, 0), (16, 3), (32, 0), (33, 70), (64, 0), (65, 1000), (129, 0), (300, 130), (515, 60)])
@pytest.mark.parametrize("name", SHAPES)
def test_prefill_shapes(name, S, P):
    _run(name, S, P)


@pytest.mark.parametrize("S", [95, 96, 97, 128, 190, 192, 193, 280])
@pytest.mark.parametrize("name", ["g128", "g64"])
def test_prefill_token_tiles(name, S):
    """Both sides of each change between tiles of 96 and 128 tokens, full and ragged last tiles."""
    _run(name, S, 5)


@pytest.mark.parametrize("offset", [1, 2, 4])
def test_prefill_value_aligned_buffers(offset):
    _run("g128", 40, 10, offset)


@pytest.mark.parametrize("name,S,P", [("g128", 3, 2000), ("g64", 17, 3000), ("g32", 70, 1500)])
def test_prefill_attention_parts(name, S, P):
    """Few token blocks over a long cache: the cache is cut into parts, some without a visible entry."""
    _run(name, S, P)
    _run(name, S, P)


@pytest.mark.parametrize("name,S", [("g128", 1), ("g64", 40), ("g128", 515)])
def test_prefill_launch_order(name, S):
    """A prefill's kernels are launched ahead of each other's ends: prompts one right after the other give the bits
    of prompts waited for, also where the second reuses the first one's buffers and row."""
    shape = SHAPES[name]
    g = GpuShard(shape, synth.make_weights(shape, 31))
    st = pkg.kv_state_alloc(g.h, 1, 2 * S)
    d_in = [to_dev(synth.hidden_in(shape, 8, i, S)) for i in range(4)]
    d_mask = to_dev(np.ones(2 * S, np.uint8))
    d_pos = [to_dev(np.arange(P, P + S, dtype=np.int32)) for P in (0, S)]
    s = torch.cuda.Stream()

    def prompts(wait):
        out = [torch.zeros_like(d_in[0]) for _ in d_in]
        torch.cuda.synchronize()
        for i, x in enumerate(d_in):  # two prompts onto the row, then two again
            if i == 2:
                pkg.kv_state_reset(st, 0)
            pkg.shard_prefill(g.h, st, 0, x.data_ptr(), None, S, d_pos[i % 2].data_ptr(), d_mask.data_ptr(),
                              (1 + i % 2) * S, out[i].data_ptr(), s.cuda_stream)
            if wait:
                pkg.shard_sync_status(g.h, s.cuda_stream)
        pkg.shard_sync_status(g.h, s.cuda_stream)
        pkg.kv_state_reset(st, 0)
        return out

    want = prompts(True)
    for _ in range(5):
        for a, b in zip(prompts(False), want):
            assert torch.equal(a, b)
    pkg.kv_state_free(st)
    g.close()
