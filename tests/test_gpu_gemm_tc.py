"""GPU parity of the many-token tensor-core projection (tcgen05,
shard_debug_gemm) against the fp64 oracle, through the C ABI: for token
counts that fill one, several and ragged token tiles, every projection of
the tiny shard (group 32), one 8B layer (group 128) and a ragged shape
(group 64, K not a multiple of 128, F not a multiple of 8) is within the
fp32 accumulation bound of the oracle; with integer activations and
power-of-two scales (every sum exact in fp32) it is bit-exact; and it
equals the decode step's GEMV where both are exact.  And as shard_prefill
launches it (shard_debug_gemm_stage): K in one to four parts, even and uneven
ones, each part's sums bit-exact; and gate|up with SwiGLU in its epilogue, F a
multiple of 32 or not."""
import numpy as np
import pytest
import torch

import oracle
import paper_2608_19147_gb300 as pkg
import synth

pytestmark = pytest.mark.gpu

SHAPES = {
    "tiny": synth.TINY,
    "8b-1layer": synth.ShardShape("8b-1layer", 1, 4096, 32, 8, 128, 14336, 128, 0.02, 0, 1e-5, 500000.0, 4096),
    "ragged": synth.ShardShape("ragged", 1, 200, 4, 4, 64, 333, 64, 0.02, 0, 1e-5, 10000.0, 256),
}


def _mats(w):
    m = w.layers[0].matrices
    return {pkg.OP_QKV: [m[0], m[1], m[2]], pkg.OP_O: [m[3]], pkg.OP_GU: [m[4], m[5]], pkg.OP_DOWN: [m[6]]}


def _gemm(h, op, x16, rows):
    S, K = x16.shape
    ld = (K + 127) // 128 * 128
    xp = np.zeros((S, ld), np.uint16)
    xp[:, :K] = x16
    dx = torch.from_numpy(xp.view(np.int16)).cuda()
    y = torch.full((S, rows), float("nan"), dtype=torch.float32, device="cuda")
    pkg.shard_debug_gemm(h, 0, op, dx.data_ptr(), ld, S, y.data_ptr(), rows, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return y.cpu().numpy().astype(np.float64)


@pytest.fixture(scope="module", params=list(SHAPES))
def shard(request):
    shape = SHAPES[request.param]
    w = synth.make_weights(shape, 99)
    h = pkg.shard_create(pkg.make_config(shape), w.layers, w.embedding)
    yield shape, w, h
    pkg.shard_destroy(h)


@pytest.mark.parametrize("S", [1, 16, 33, 128, 300])
def test_gemm_matches_oracle(shard, S):
    shape, w, h = shard
    rng = np.random.default_rng(S)
    mats = _mats(w)
    for op in range(4):
        rows, K, _ = pkg.shard_debug_op_info(h, 0, op)
        x16 = rng.standard_normal((S, K)).astype(np.float16)
        got = _gemm(h, op, x16.view(np.uint16), rows)
        want = np.concatenate([oracle.gemv(m, x16.astype(np.float64)) for m in mats[op]], axis=1)
        scale = np.abs(x16.astype(np.float64)) @ np.abs(np.concatenate([oracle.dequant(m) for m in mats[op]])).T
        assert np.isfinite(got).all(), op
        assert np.all(np.abs(got - want) <= 1e-5 * scale + 1e-6), (op, np.max(np.abs(got - want) / (scale + 1e-9)))


def test_gemm_integer_inputs_bit_exact_and_equal_to_the_gemv():
    shape = SHAPES["8b-1layer"]
    rng = np.random.default_rng(5)
    w = synth.make_weights(shape, 5)
    for lw in w.layers:
        for m in lw.matrices:
            m.scales[:] = rng.choice(np.array([2.0 ** -3, 2.0 ** -4], dtype=np.float16).view(np.uint16), m.scales.shape)
    h = pkg.shard_create(pkg.make_config(shape), w.layers, w.embedding)
    try:
        mats = _mats(w)
        for op in range(4):
            rows, K, _ = pkg.shard_debug_op_info(h, 0, op)
            x16 = rng.integers(-4, 5, (40, K)).astype(np.float16)
            got = _gemm(h, op, x16.view(np.uint16), rows)
            want = np.concatenate([oracle.gemv(m, x16.astype(np.float64)) for m in mats[op]], axis=1)
            assert np.array_equal(got, want), op
            dx = torch.from_numpy(x16[:16].view(np.int16)).cuda()
            y = torch.empty((16, rows), dtype=torch.float32, device="cuda")
            pkg.shard_debug_gemv(h, 0, op, dx.data_ptr(), 16, y.data_ptr(), rows,
                                 torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            assert np.array_equal(y.cpu().numpy().astype(np.float64), got[:16]), op
    finally:
        pkg.shard_destroy(h)


# upr (units of 128 inputs) of q|k|v, o, gate|up, down: 5, 4, 5, 9 / 5, 2, 5, 3
STAGE_SHAPES = {
    "uneven": synth.ShardShape("uneven", 1, 640, 8, 2, 64, 1100, 128, 0.02, 0, 1e-5, 10000.0, 256),
    "ragged-f": synth.ShardShape("ragged-f", 1, 616, 4, 4, 64, 333, 64, 0.02, 0, 1e-5, 10000.0, 256),
    "g32": synth.ShardShape("g32", 1, 640, 8, 8, 64, 1024, 32, 0.02, 0, 1e-5, 10000.0, 256),
}


def _stage_order(x):
    """Inputs of each block of 32 to the kernel's positions; zero-padded to a multiple of 128."""
    S, K = x.shape
    p = np.zeros((S, (K + 127) // 128 * 128), x.dtype)
    k = np.arange(K)
    p[:, (k & ~31) + 16 * ((k >> 2) & 1) + 4 * ((k >> 3) & 3) + (k & 3)] = x
    return p


@pytest.fixture(scope="module", params=list(STAGE_SHAPES))
def stage(request):
    shape = STAGE_SHAPES[request.param]
    w = synth.make_weights(shape, 7)
    rng = np.random.default_rng(7)
    for m in w.layers[0].matrices:  # sums of integers times 2^-8 or 2^-9: exact in fp32
        m.scales[:] = rng.choice(np.array([2.0 ** -8, 2.0 ** -9], dtype=np.float16).view(np.uint16), m.scales.shape)
    h = pkg.shard_create(pkg.make_config(shape), w.layers, w.embedding)
    yield shape, w, h
    pkg.shard_destroy(h)


@pytest.mark.parametrize("S", [1, 40, 77, 130])
def test_stage_gemm_parts_bit_exact(stage, S):
    shape, w, h = stage
    rng = np.random.default_rng(S)
    for op, mats in _mats(w).items():
        rows, K, _ = pkg.shard_debug_op_info(h, 0, op)
        x = rng.integers(-4, 5, (S, K)).astype(np.float16)
        xp = _stage_order(x.view(np.uint16))
        dx = torch.from_numpy(xp.view(np.int16)).cuda()
        dense = np.concatenate([oracle.dequant(m) for m in mats])
        upr = xp.shape[1] // 128
        for parts in range(0, min(4, upr) + 1):
            y = torch.full((4, S, rows), float("nan"), dtype=torch.float32, device="cuda")
            n = pkg.shard_debug_gemm_stage(h, 0, op, dx.data_ptr(), xp.shape[1], S, parts, y=y.data_ptr(), y_ld=rows,
                                           y_part=S * rows, stream=torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            assert n == parts or (parts == 0 and 1 <= n <= 4)
            got = y.cpu().numpy().astype(np.float64)
            for p in range(n):  # part p: units [upr p / n, upr (p + 1) / n)
                k = slice(128 * (upr * p // n), min(K, 128 * (upr * (p + 1) // n)))
                assert np.array_equal(got[p], x[:, k].astype(np.float64) @ dense[:, k].T), (op, parts, p)
            assert np.isnan(got[n:]).all()


@pytest.mark.parametrize("S", [1, 40, 77, 130])
def test_stage_gemm_swiglu(stage, S):
    shape, w, h = stage
    F = shape.ffn
    rng = np.random.default_rng(S)
    x = rng.integers(-4, 5, (S, shape.hidden)).astype(np.float16)
    xp = _stage_order(x.view(np.uint16))
    dx = torch.from_numpy(xp.view(np.int16)).cuda()
    ld = (F + 127) // 128 * 128 + 8
    hd = torch.full((S + 1, ld), 0x5555, dtype=torch.int16, device="cuda")
    assert pkg.shard_debug_gemm_stage(h, 0, pkg.OP_GU, dx.data_ptr(), xp.shape[1], S, h=hd.data_ptr(), h_ld=ld,
                                      stream=torch.cuda.current_stream().cuda_stream) == 1
    torch.cuda.synchronize()
    raw = hd.cpu().numpy().view(np.uint16)
    j = np.arange(F)
    at = (j & ~31) + 16 * ((j >> 2) & 1) + 4 * ((j >> 3) & 3) + (j & 3)
    assert (np.delete(raw[:S], at, axis=1) == 0x5555).all() and (raw[S] == 0x5555).all()  # past F, and the next row
    gate, up = [x.astype(np.float64) @ oracle.dequant(m).T for m in w.layers[0].matrices[4:6]]
    want = gate / (1 + np.exp(-gate)) * up
    got = raw[:S][:, at].view(np.float16).astype(np.float64)
    # gate and up are exact; silu in fp32 (expf, one addition, one division, one product: under 8 units of 2^-24)
    # and one rounding to fp16 (half a unit of 2^-10 of the power of two below, 2^-25 among subnormals)
    assert (np.abs(got - want) <= np.abs(want) * (2.0 ** -11 + 2.0 ** -21) + 2.0 ** -25).all()


def test_stage_gemm_refuses_what_it_cannot_do(stage):
    shape, w, h = stage
    x = torch.zeros((1, 1280), dtype=torch.int16, device="cuda")
    y = torch.zeros((8, 8192), dtype=torch.float32, device="cuda")
    for kw in (dict(parts=5, y=y.data_ptr(), y_ld=4096, y_part=4096), dict(parts=2, h=y.data_ptr(), h_ld=2048),
               dict(parts=1), dict(parts=1, y=y.data_ptr(), y_ld=4, y_part=4096)):
        with pytest.raises(pkg.ShardError):
            pkg.shard_debug_gemm_stage(h, 0, pkg.OP_GU, x.data_ptr(), 1280, 1, **kw)
    # K of o is 512 or 256: no more parts than units of 128 inputs
    with pytest.raises(pkg.ShardError):
        pkg.shard_debug_gemm_stage(h, 0, pkg.OP_O, x.data_ptr(), 1280, 1, parts=shape.n_heads * 64 // 128 + 1, y=y.data_ptr(),
                                   y_ld=4096, y_part=4096)
