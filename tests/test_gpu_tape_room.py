"""The kill tape of a launch-per-factor gradient where one cut drops more than a
page of it (2^20 records): energies within 1e-10 Ha, gradients within 1e-8 of the
same evaluation on a context whose tape grew with its table.
"""
import dataclasses

import numpy as np
import pytest

from paper_2301_05726_gb300 import synth

pytestmark = pytest.mark.gpu
E_TOL = 1e-10
G_TOL = 1e-8


@pytest.mark.parametrize("stride", [0, 20])
def test_a_cut_of_more_than_a_page(stride):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_05726_gb300 import build
    build.build()
    from paper_2301_05726_gb300.api import UCCContext
    # Singles of distinct electrons into distinct orbitals: each doubles the table.  The last
    # one leaves 2^21 entries, of which 1,000 stay.
    rng = np.random.default_rng(5)
    h, g = synth.make_integrals(rng, 22)
    rows = [(2 * i + s, -1, 2 * (i + 11) + s, -1) for s in (0, 1) for i in range(11)][:21]
    p = synth.Problem(22, 11, 11, h, g, np.array(rows, dtype=np.int32), rng.uniform(0.15, 0.35, 21), eps=0.0)
    p = dataclasses.replace(p, n_max=1_200_000, n_cut=1000)
    ctx, fresh = UCCContext(p), UCCContext(p)
    for c in (ctx, fresh):
        c.set_options(probe_width=1, checkpoint_stride=stride)  # a launch per factor
    ctx.apply()  # its table has its full size before the gradient: no growth makes room on the tape
    E, grad = ctx.gradient()
    Er, gr = fresh.gradient()
    assert ctx.stats()["tape_entries"] >= (1 << 21) - 1000
    assert abs(E - Er) <= E_TOL and np.max(np.abs(grad - gr)) <= G_TOL
