"""Resident passes (a whole run of factors in one launch, the table in the
shared memory of a thread-block cluster or of the whole GPU) against the
launch-per-factor kernels and the CPU oracle: the same determinants and bit-identical amplitudes, counts, entropies
(1e-10), energies (1e-10 Ha) and gradients (1e-8).

The shapes sit where the resident kernels change behaviour: every cluster size,
tables below and above one thread per entry, heavy eps drops with revivals,
cuts that keep one entry or all but a few, ties larger than the ranked
candidate list (also on the key's words), two-word keys, tables just above the
clusters' size and of the whole GPU's, a table that outgrows the GPU's shared
memory on the way, and a tape that needs more than one launch.
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


def problem(name):
    def make(n, a, b, eps=0.0, cut=(0, 0), pre=None, zero_from=None, sigma=0.08, md=None):
        p = synth.make_problem(77, n, a, b, sigma, eps=eps, m_doubles=md, name=name)
        if pre:
            p = p.prefix(pre)
        if zero_from is not None:
            th = p.theta.copy()
            th[zero_from:] = 0.0
            p = p.with_theta(th)
        p.n_max, p.n_cut = cut
        return p

    return {
        "one_cta": lambda: make(5, 2, 1),
        "one_cta_open_shell_eps": lambda: make(6, 3, 2, eps=1e-4),
        "four_ctas": lambda: make(7, 3, 2),
        "eight_ctas": lambda: make(8, 4, 3, eps=1e-7),
        "sixteen_ctas": lambda: make(9, 3, 3),
        "drops_and_revivals": lambda: make(9, 3, 3, eps=1e-2, sigma=0.3),
        "cut_keeps_all": lambda: make(9, 3, 3, cut=(1000, 1000)),
        "cut_keeps_one": lambda: make(8, 3, 3, cut=(40, 1), pre=200),
        "cut_odd": lambda: make(10, 4, 3, eps=1e-6, cut=(2999, 1701), pre=500),
        "ties": lambda: make(9, 4, 4, cut=(5000, 4001), pre=260, zero_from=8),
        "ties_wide": lambda: make(36, 3, 3, cut=(3000, 2501), pre=200, zero_from=8),
        "wide_eps_cut": lambda: make(40, 4, 3, eps=1e-6, cut=(1601, 1000), pre=250),
        "grid": lambda: make(12, 4, 4, pre=260),
        "grid_drops_and_revivals": lambda: make(11, 4, 3, eps=1e-4, sigma=0.2, pre=400),
        "grid_cut": lambda: make(14, 4, 4, eps=1e-9, cut=(30001, 17001), pre=220),
        "grid_ties": lambda: make(12, 4, 4, cut=(20000, 16001), pre=220, zero_from=8),
        "grid_ties_wide": lambda: make(36, 3, 3, cut=(20000, 16001), pre=330, zero_from=8),
        "grid_wide": lambda: make(34, 3, 3, eps=1e-7, cut=(24000, 15000), pre=260),
    }[name]()


CASES = ["one_cta", "one_cta_open_shell_eps", "four_ctas", "eight_ctas", "sixteen_ctas", "drops_and_revivals",
         "cut_keeps_all", "cut_keeps_one", "cut_odd", "ties", "ties_wide", "wide_eps_cut", "grid",
         "grid_drops_and_revivals", "grid_cut", "grid_ties", "grid_ties_wide", "grid_wide"]


def same_state(got, want):
    assert np.array_equal(got[0], want[0])
    assert not np.any(got[1] != want[1])


@pytest.mark.parametrize("name", CASES)
def test_state_and_gradient(torch_cuda, name):
    import oracle
    from paper_2301_05726_gb300.api import UCCContext
    p = problem(name)
    o = oracle.Oracle(p)
    ok, oa, oc = o.apply()
    E_o, g_o = o.gradient()
    ctx = UCCContext(p)
    ctx.apply()
    st = ctx.stats()
    same_state(ctx.wavefunction(), (ok, oa))
    for c in ("rotations", "created", "dropped_new", "dropped_old", "cut"):
        assert st[c] == oc[c], c
    assert st["forward_launches"] == 1  # the resident path ran
    E, g = ctx.gradient()
    assert abs(E - E_o) <= E_TOL and np.max(np.abs(g - g_o)) <= G_TOL
    general = UCCContext(p)
    general.set_options(rebuild_test_regions=1)  # launch per factor
    general.apply()
    assert general.stats()["forward_launches"] >= p.n_exc
    same_state(general.wavefunction(), (ok, oa))
    Eg, gg = general.gradient()
    assert abs(E - Eg) <= E_TOL and np.max(np.abs(g - gg)) <= G_TOL


@pytest.mark.parametrize("name", ["cut_odd", "wide_eps_cut", "grid_cut", "grid_ties"])
def test_cut_threshold_that_moves(torch_cuda, name):
    """Angles whose size changes by powers of ten on the way: a cut's threshold
    lies near the last one's, below its window, above it, or in a bin of ties."""
    import oracle
    from paper_2301_05726_gb300.api import UCCContext
    p = problem(name)
    scale = np.array([1.0, 1e-3, 1.0, 10.0, 1e-6])[np.arange(p.n_exc) * 5 // p.n_exc]
    p2 = p.with_theta(np.clip(p.theta * scale, -0.7, 0.7))
    p2.n_max, p2.n_cut = p.n_max, p.n_cut
    ok, oa, oc = oracle.Oracle(p2).apply()
    ctx = UCCContext(p2)
    ctx.apply()
    st = ctx.stats()
    same_state(ctx.wavefunction(), (ok, oa))
    for c in ("rotations", "created", "dropped_new", "dropped_old", "cut"):
        assert st[c] == oc[c], c
    assert st["forward_launches"] == 1 and oc["cut"] > 0


@pytest.mark.parametrize("name", ["one_cta_open_shell_eps", "sixteen_ctas", "cut_odd", "grid_cut"])
def test_entropy(torch_cuda, name):
    import oracle
    from paper_2301_05726_gb300.api import UCCContext
    p = problem(name)
    ctx = UCCContext(p)
    ctx.set_options(record_entropy=1)
    ctx.apply()
    S = oracle.Oracle(p).entropy_per_factor(n_max=p.n_max, n_cut=p.n_cut)
    assert np.max(np.abs(ctx.entropy() - S)) <= 1e-10


@pytest.mark.parametrize("name", ["one_cta", "drops_and_revivals", "wide_eps_cut", "grid_drops_and_revivals"])
def test_entropy_of_revived_entries(torch_cuda, name):
    """The kept terms of entries that are dropped, come back, move in a
    compaction or are cut."""
    import oracle
    from paper_2301_05726_gb300.api import UCCContext
    p = problem(name)
    ctx = UCCContext(p)
    ctx.set_options(record_entropy=1)
    ctx.apply()
    assert ctx.stats()["forward_launches"] == 1
    S = oracle.Oracle(p).entropy_per_factor(n_max=p.n_max, n_cut=p.n_cut)
    assert np.max(np.abs(ctx.entropy() - S)) <= 1e-10


def test_outgrows_the_gpu(torch_cuda):
    # Resident to begin with; past some 700,000 determinants a launch per factor.
    from paper_2301_05726_gb300.api import UCCContext
    p = synth.make_problem(77, 15, 4, 4, 0.08).prefix(900)
    ctx, general = UCCContext(p), UCCContext(p)
    general.set_options(rebuild_test_regions=1)
    for c in (ctx, general):
        c.apply()
    st, sg = ctx.stats(), general.stats()
    assert 1 < st["forward_launches"] < sg["forward_launches"] and st["n_det"] > 900_000
    for c in ("n_det", "rotations", "created"):
        assert st[c] == sg[c], c
    same_state(ctx.wavefunction(), general.wavefunction())
    E, g = ctx.gradient()
    Eg, gg = general.gradient()
    assert abs(E - Eg) <= E_TOL and np.max(np.abs(g - gg)) <= G_TOL


@pytest.mark.parametrize("name,pre,stride", [("cut_odd", 150, 1), ("cut_odd", 150, 37), ("grid_cut", 120, 11)])
def test_segments(torch_cuda, name, pre, stride):
    # Checkpointed gradients run each segment resident, forward and reverse.
    import oracle
    from paper_2301_05726_gb300.api import UCCContext
    whole = problem(name)
    p = whole.prefix(pre)
    p.n_max, p.n_cut = whole.n_max, whole.n_cut
    ctx = UCCContext(p)
    ctx.set_options(checkpoint_stride=stride)
    E, g = ctx.gradient()
    E_o, g_o = oracle.Oracle(p).gradient()
    assert abs(E - E_o) <= E_TOL and np.max(np.abs(g - g_o)) <= G_TOL


def test_tape_of_several_pages(torch_cuda):
    # More records than a page of 2^20 holds: the first launch stops for tape,
    # the next goes on.
    from paper_2301_05726_gb300.api import UCCContext
    p = synth.fig3_problem().prefix(1000)
    p.n_max, p.n_cut = 8000, 5000
    ctx = UCCContext(p)
    E, g = ctx.gradient()
    st = ctx.stats()
    assert st["tape_entries"] > (1 << 20) and 1 < st["forward_launches"] < 20
    E2, g2 = ctx.gradient()  # the pages are there now
    assert ctx.stats()["forward_launches"] == 1
    ctx.set_options(rebuild_test_regions=1)
    Eg, gg = ctx.gradient()
    for e, d in ((E, g), (E2, g2)):
        assert abs(e - Eg) <= E_TOL and np.max(np.abs(d - gg)) <= G_TOL


def test_batch_mixes_cluster_sizes_and_paths(torch_cuda):
    # Jobs of every size share a launch; a job too large for a cluster and a
    # two-word one take their own paths in the same call.
    from paper_2301_05726_gb300.api import UCCContext, batch_run
    names = ["one_cta", "cut_odd", "eight_ctas", "grid", "ties", "wide_eps_cut", "cut_keeps_one", "four_ctas",
             "sixteen_ctas", "drops_and_revivals", "one_cta_open_shell_eps", "cut_keeps_all"]
    probs = [problem(n) for n in names]
    ctxs = [UCCContext(p) for p in probs]
    E, grads = batch_run(ctxs, 1e-7, with_grad=True)
    for n, p, e, g in zip(names, probs, E, grads):
        ref = UCCContext(p)
        ref.set_options(rebuild_test_regions=1)
        Er, gr = ref.gradient(eps=1e-7)
        assert abs(e - Er) <= E_TOL and np.max(np.abs(g - gr)) <= G_TOL, n


@pytest.mark.parametrize("eps,sigma,angles", [
    (2.0 ** -12, 0.3, None), (2.0 ** -7, 0.5, None), (1e-6, 0.05, None), (0.02, 1.5, None),
    (5e-324, 0.1, None), (1e-300, 0.1, None),
    (2.0 ** -10, 0.1, "exact"), (1e-4, 0.1, "zeros")])
def test_launch_per_factor_settles_lone_entries_exactly(torch_cuda, eps, sigma, angles):
    # A launch per factor settles lone entries by the exponents of their
    # amplitude and sin(theta): thresholds that are powers of two, products that
    # fall on them, zero angles, large angles, thresholds below every normal
    # number; counts and amplitudes bit for bit, and the gradient.
    import oracle
    from paper_2301_05726_gb300.api import UCCContext
    p = synth.make_problem(5, 8, 3, 3, sigma, eps=eps).prefix(260)
    th = p.theta.copy()
    if angles == "exact":
        th[::3] = np.arcsin(2.0 ** -5)  # products 2^-5 2^-5 on the threshold 2^-10
    elif angles == "zeros":
        th[1::2] = 0.0
    p = p.with_theta(th)
    p.eps = eps
    ok, oa, oc = oracle.Oracle(p).apply()
    E_o, g_o = oracle.Oracle(p).gradient()
    ctx = UCCContext(p)
    ctx.set_options(rebuild_test_regions=1)
    ctx.apply()
    st = ctx.stats()
    same_state(ctx.wavefunction(), (ok, oa))
    for c in ("rotations", "created", "dropped_new", "dropped_old"):
        assert st[c] == oc[c], c
    E, g = ctx.gradient()
    assert abs(E - E_o) <= E_TOL and np.max(np.abs(g - g_o)) <= G_TOL
    res = UCCContext(p)  # the resident path takes the same decisions
    res.apply()
    same_state(res.wavefunction(), (ok, oa))
