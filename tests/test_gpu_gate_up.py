"""The step's gate|up projection for every token count of a step: sums reduced
in the CTA's shared memory (a slot per warp and token) give each request's row
the same bits as the row alone, and match the oracle at the fixed bar, for
row-blocks split over 2, 4 and 12 warps and a ragged last row-block."""
import numpy as np
import pytest

import oracle
import synth
from gpu_engine import GpuEngine, GpuShard, assert_close

pytestmark = pytest.mark.gpu

SHAPES = {
    "g32": synth.ShardShape("g32", 1, 256, 4, 2, 64, 688, 32, 0.02, 0, 1e-5, 10000.0, 64),
    "g64-ragged": synth.ShardShape("g64", 1, 520, 4, 4, 64, 333, 64, 0.02, 0, 1e-5, 10000.0, 64),
    "g128-long-k": synth.ShardShape("g128", 1, 3072, 2, 1, 128, 1000, 128, 0.02, 0, 1e-5, 10000.0, 64),
}


@pytest.mark.parametrize("name", SHAPES)
def test_gate_up_rows(name):
    shape = SHAPES[name]
    w = synth.make_weights(shape, 21)
    g = GpuShard(shape, w)
    h = synth.hidden_in(shape, 22, 0, 16)
    ref = oracle.OracleShard(shape, w)

    def step(eng, rows):
        n = len(rows)
        return eng.step([1] * n, np.zeros(n, np.int32), np.ones((n, 4), np.uint8), hidden_in=h[rows])

    alone, single = GpuEngine(g, 1, 4), []
    for r in range(16):
        single.append(step(alone, [r]))
        alone.trim(0, np.zeros(1, np.uint8))  # empty again
    single = np.concatenate(single)
    for M in (2, 5, 6, 8, 9, 11, 16):
        eng, o = GpuEngine(g, M, 4), ref.state(M, 4)
        got = step(eng, list(range(M)))
        rc, want, _ = o.step([1] * M, np.zeros(M, np.int32), np.ones((M, 4), np.uint8), hidden_in=h[:M])
        assert rc == 0
        assert_close(got, want, what="%s M=%d" % (name, M))
        assert np.array_equal(got, single[:M]), (name, M)
        eng.close()
    alone.close()
    g.close()
