"""Several contexts alive at once.

Kernels are shared between contexts whose launches differ in size: how much shared memory a block takes
depends on the weight quantizer (the l2 term's held weights come with a tile's stage) and on the worker count.
What one context sets up must not take anything from another's launches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

import paper_2004_14180_b200 as qb  # noqa: E402
from _parity import Pair  # noqa: E402

S_MODE, W_MODE = qb.PLACE_SERVER, qb.PLACE_WORKER
STREAM = qb.QAdamOptions(worker_kernel=qb.WORKER_STREAMING)
DECAY = 5e-4


# (kg, grid, placement, decay, options) and, for either context, (kx, n)
@pytest.mark.parametrize("kg,grid,placement,decay,options,one,two", [
    (0, 0, S_MODE, DECAY, STREAM, (6, 2), (-1, 2)),       # sweep and its settle pass
    (0, 0, S_MODE, DECAY, STREAM, (0, 2), (14, 2)),
    (1, 0, S_MODE, DECAY, STREAM, (6, 2), (14, 2)),
    (3, 1, S_MODE, DECAY, STREAM, (6, 2), (-1, 2)),       # first pass that only reads
    (3, 1, W_MODE, DECAY, STREAM, (14, 2), (6, 2)),       # first pass with the moments
    (0, 0, S_MODE, DECAY, None, (6, 2), (0, 2)),          # on chip
    (0, 0, W_MODE, DECAY, None, (14, 2), (-1, 2)),
    (0, 0, S_MODE, 0.0, None, (0, 5), (0, 7)),            # pipelined server pass, worker count at run time
    (3, 1, S_MODE, 0.0, None, (0, 3), (0, 50)),
    (6, 1, S_MODE, 0.0, None, (0, 65), (0, 100)),         # plain server pass, a table per worker
])
@pytest.mark.parametrize("swap", [False, True])
def test_two_contexts_stepped_in_turn(kg, grid, placement, decay, options, one, two, swap):
    # Either order of creation, and a third context that comes and goes in between.  Launches are counted: a
    # refused on-chip launch would otherwise hide behind the streaming ones that take its place.
    rng = np.random.default_rng(10 * kg + one[0])
    seg = [4096 + 130, 700, 2 * 4096]
    d = sum(seg)

    def make(kx, n):
        p = Pair(seg, n, kg, kx, placement, x1=(rng.standard_normal(d) * 0.2).astype(np.float32), grid_g=grid,
                 options=options)
        p.set_regularization(decay)
        return p

    pairs = [make(*c) for c in ((two, one) if swap else (one, two))]
    before = [p.gpu.launches for p in pairs]
    for t in range(2):
        for p in pairs:
            p.step((rng.standard_normal((p.gpu.n, d)) * 0.01).astype(np.float32))
            p.compare_state()
        if t == 0:
            make(*two).close()
            make(*one).close()
    per_step = 3 if options is STREAM else 2
    assert [p.gpu.launches - b for p, b in zip(pairs, before)] == [2 * per_step] * 2
    for p in pairs:
        p.close()
