"""The bucketed energy's pair walk at the sizes where it changes behaviour: core
groups larger than a block's shared memory (walked in global memory), partitions
taken bin range by bin range, empty cores (two electrons), open shells, and
two-word keys; against the per-connection route (the same pairs, sigma to
rounding) and the CPU oracle (1e-10 Ha)."""
import numpy as np
import pytest

from paper_2301_05726_gb300 import synth
from test_gpu_energy_buckets import assert_routes_agree, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


# n_spatial, n_alpha, n_beta, partitions (0: the library's choice)
SHAPES = [
    (48, 1, 1, 0),   # one double core, empty, of 2,304 records; two-word keys
    (32, 1, 1, 1),   # the same in one word, 1,024 records
    (40, 2, 1, 2),   # 7,203 records in two partitions
    (7, 3, 3, 1),    # 18,375 records in one partition
    (7, 4, 2, 8),
    (9, 1, 3, 0),
    (6, 2, 2, 64),   # fewer records than bins
]


@pytest.mark.parametrize("n,a,b,partitions", SHAPES)
def test_pair_walk(torch_cuda, n, a, b, partitions):
    import oracle
    from paper_2301_05726_gb300.api import UCCContext
    p = synth.make_problem(n, n, a, b, 0.1)
    if p.n_exc > 2400:
        p = p.prefix(2400)
    ctx = UCCContext(p)
    ctx.apply()
    E = assert_routes_agree(ctx, partitions=partitions)
    o = oracle.Oracle(p)
    k, amps, _ = o.apply()
    E_o, _ = o.energy(k, amps)
    assert len(k) == ctx.stats()["n_det"] and abs(E - E_o) <= 1e-10
    assert np.isfinite(E)
