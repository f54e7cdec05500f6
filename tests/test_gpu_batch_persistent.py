"""The persistent batch kernels and the cuts on the device inside them.  Batches whose
jobs all fit a thread-block cluster run resident; batch_tiles keeps these in the
persistent launches.  Amplitudes bit for bit with the oracle, energies within 1e-10 Ha,
gradients within 1e-8 of a launch per factor with host-driven cuts.
"""
import numpy as np
import pytest

from paper_2301_05726_gb300 import synth

pytestmark = pytest.mark.gpu
E_TOL = 1e-10
G_TOL = 1e-8


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_05726_gb300 import build
    build.build()
    return torch


def job(j, prefix=None):
    p = synth.batch_job_problem(j)
    p = p.prefix(prefix) if prefix else p
    p.n_max, p.n_cut = 8000, 5000
    return p


def contexts(probs, **options):
    from paper_2301_05726_gb300.api import UCCContext
    out = [UCCContext(p) for p in probs]
    for c in out:
        c.set_options(**options)
    return out


@pytest.mark.parametrize("tiles", [1, 2, 8])
def test_cut_jobs_state_vs_oracle(torch_cuda, tiles):
    import oracle
    from paper_2301_05726_gb300.api import batch_run
    probs = [job(54, 300), job(120, 300), job(0)]
    ctxs = contexts(probs, batch_tiles=tiles)
    E, _ = batch_run(ctxs, eps=1e-8, with_grad=False)
    assert ctxs[0].stats()["batch_tiles"] == tiles
    for p, c, e in zip(probs, ctxs, E):
        o = oracle.Oracle(p)
        ok, oa, oc = o.apply(eps=1e-8)
        gk, ga = c.wavefunction()
        assert np.array_equal(gk, ok) and not np.any(ga != oa), p.name
        assert c.stats()["cut"] == oc["cut"] and c.stats()["rotations"] == oc["rotations"], p.name
        assert abs(e - o.energy(ok, oa)[0]) <= E_TOL, p.name
    assert sum(c.stats()["cut"] > 0 for c in ctxs) == 2


def test_gradients_vs_a_launch_per_factor(torch_cuda):
    from paper_2301_05726_gb300.api import batch_run
    probs = [job(j) for j in (0, 3, 21, 54, 65, 98, 120, 131, 186, 197, 230, 251)]
    ctxs = contexts(probs, batch_tiles=2)
    E, grads = batch_run(ctxs, eps=1e-8, with_grad=True)
    assert ctxs[0].stats()["batch_tiles"] == 2
    cut_jobs = 0
    for p, c, e, g, ref in zip(probs, ctxs, E, grads, contexts(probs, rebuild_test_regions=1)):
        Er, gr = ref.gradient(eps=1e-8)
        assert abs(e - Er) <= E_TOL and np.max(np.abs(g - gr)) <= G_TOL, p.name
        assert ref.stats()["forward_launches"] >= p.n_exc
        assert c.stats()["cut"] == ref.stats()["cut"], p.name
        cut_jobs += ref.stats()["cut"] > 0
    assert cut_jobs >= 4
