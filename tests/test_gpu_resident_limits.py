"""Where a resident pass meets a limit -- an inbox, its room, the tape, memory, a
wait -- the call gives what a launch per factor gives: energies within 1e-10 Ha,
gradients within 1e-8, and the same determinants, amplitudes and counts.
"""
import dataclasses

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


def doubling(n_factors, extra=(), n=20):
    """Singles of distinct electrons into distinct orbitals, half of them filled, so that every factor
    doubles the table, then the rows of extra."""
    half = n // 2
    rng = np.random.default_rng(5)
    h, g = synth.make_integrals(rng, n)
    rows = [(2 * i + s, -1, 2 * (i + half) + s, -1) for s in (0, 1) for i in range(half)][:n_factors]
    exc = np.array(rows + list(extra), dtype=np.int32)
    return synth.Problem(n, half, half, h, g, exc, rng.uniform(0.15, 0.35, len(exc)), eps=0.0)


def context(p, **options):
    from paper_2301_05726_gb300.api import UCCContext
    c = UCCContext(p)
    c.set_options(**options)
    return c


def assert_gradient(got, p, **options):
    E, g = got
    Er, gr = context(p, rebuild_test_regions=1, **options).gradient()  # a launch per factor
    assert abs(E - Er) <= E_TOL and np.max(np.abs(g - gr)) <= G_TOL


@pytest.mark.parametrize("n_cut", [100_000, 350_000])
def test_reverse_meets_a_cut_larger_than_the_inboxes(torch_cuda, n_cut):
    # The cut after the last single drops more determinants than the GPU's inboxes
    # take together (or than they take beside the messages of the factor after it),
    # while the final state is small.
    p = doubling(20, extra=[(0, 1, 20, 21), (2, 3, 22, 23)])
    p = dataclasses.replace(p, n_max=1_000_000, n_cut=n_cut)
    ctx = context(p)
    assert_gradient(ctx.gradient(), p)
    assert ctx.stats()["cut"] >= (1 << 20) - n_cut


def test_problems_of_several_sizes_in_several_threads(torch_cuda):
    # Launches of one kernel with more and with less shared memory, from threads of their own.
    import threading
    big = dataclasses.replace(synth.fig3_problem().prefix(3), n_max=8000, n_cut=5000)
    small = synth.make_problem(77, 9, 3, 3, 0.08).prefix(3)
    errors = []

    def work(p, runs):
        try:
            with torch_cuda.cuda.stream(torch_cuda.cuda.Stream()):
                c = context(p)
                for _ in range(runs):
                    c.apply()
        except Exception as e:  # the thread's failure is the test's
            errors.append(e)

    threads = [threading.Thread(target=work, args=(p, 2000)) for p in (big, small, small, big)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


def test_the_whole_gpu_serves_a_sector_of_any_size(torch_cuda):
    # 3.6e17 determinants in the sector: the room is the GPU's, not the sector's.
    p = doubling(17, n=32)
    ctx, general = context(p), context(p, rebuild_test_regions=1)
    for c in (ctx, general):
        c.apply()
    assert ctx.stats()["n_det"] == 1 << 17 and ctx.stats()["forward_launches"] == 1
    for x, y in zip(ctx.wavefunction(), general.wavefunction()):
        assert np.array_equal(x, y)


def test_a_segment_that_starts_without_room(torch_cuda):
    # 2^19 determinants at the end of a resident segment; the next one's only factor
    # doubles them, past the resident room and past the table's capacity.
    p = doubling(20)
    ctx = context(p, checkpoint_stride=19)
    assert_gradient(ctx.gradient(), p, checkpoint_stride=19)
    assert ctx.stats()["n_det"] == 1 << 20


@pytest.mark.parametrize("options", [dict(checkpoint_stride=100, tape_budget_mb=100), dict(tape_budget_mb=48)])
def test_a_tape_that_fits_the_launches_but_not_full_tables(torch_cuda, options):
    # Some 250,000 records in all, 140,000 in a segment (a page of 24 MiB); a resident
    # pass over a table of this size wants ten times as many at once.
    p = synth.make_problem(77, 15, 4, 4, 0.02, eps=1e-6).prefix(400)
    ctx, general = context(p, **options), context(p, rebuild_test_regions=1, **options)
    E, g = ctx.gradient()
    Er, gr = general.gradient()
    assert abs(E - Er) <= E_TOL and np.max(np.abs(g - gr)) <= G_TOL
    st, sg = ctx.stats(), general.stats()
    for x in ("tape_entries", "created", "dropped_old", "recompute_rotations"):
        assert st[x] == sg[x], x


@pytest.mark.parametrize("left_mb", [44, 84, 120])
def test_less_memory_than_a_resident_pass_wants(torch_cuda, left_mb):
    # A resident gradient over this sector wants a table of 66 MB, for what it may
    # write back, inboxes of 41 MB and 240 MB of tape; 14,841 determinants
    # take some 5 MB, and a launch per factor one page of tape, 24 MiB.
    torch = torch_cuda
    p = synth.make_problem(77, 15, 4, 4, 0.05).prefix(60)
    options = dict(energy_route=1)  # the bucketed energy's buffers have their own fallback
    for more in (dict(), dict(rebuild_test_regions=1)):
        context(p, **options, **more).gradient()  # every kernel is loaded
    ctx = context(p, **options)
    hold = []
    try:
        torch.cuda.synchronize()
        for step in (1 << 30, 1 << 24, 1 << 21):
            while torch.cuda.mem_get_info()[0] > (left_mb << 20) + step:
                n = (torch.cuda.mem_get_info()[0] - (left_mb << 20)) // step * step
                hold.append(torch.empty(n, dtype=torch.uint8, device="cuda"))
        ctx.apply()
        E, g = ctx.gradient()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert ctx.stats()["forward_launches"] >= p.n_exc  # no resident pass
    assert_gradient((E, g), p, **options)


@pytest.mark.parametrize("wide", [False, True])
def test_a_wait_that_runs_out(torch_cuda, wide):
    # A block of every whole-GPU launch leaves before its first barrier (a test hook),
    # so the others' waits run out after 50 ms: a launch per factor takes over.
    p = (synth.make_problem(77, 34, 3, 3, 0.08, eps=1e-7).prefix(120) if wide
         else synth.make_problem(77, 12, 4, 4, 0.08).prefix(120))
    if wide:
        p.n_max, p.n_cut = 24000, 15000
    hook = dict(batch_wait_ms=50, batch_test_skip_block=2)
    ctx, general = context(p, **hook), context(p, rebuild_test_regions=1)
    for c in (ctx, general):
        c.apply()
    assert ctx.stats()["forward_launches"] > p.n_exc  # the one that gave up, and one per factor
    for x, y in zip(ctx.wavefunction(), general.wavefunction()):
        assert np.array_equal(x, y)
    assert_gradient(ctx.gradient(), p)
    assert_gradient(context(p, checkpoint_stride=25, **hook).gradient(), p)
    entropies = []
    for options in (hook, dict(rebuild_test_regions=1)):
        c = context(p, record_entropy=1, **options)
        c.apply()
        entropies.append(c.entropy())
    assert np.max(np.abs(entropies[0] - entropies[1])) <= 1e-10
    ctx.set_options(batch_wait_ms=0, batch_test_skip_block=0)  # the same context runs resident again
    ctx.apply()
    assert ctx.stats()["forward_launches"] == 1
    for x, y in zip(ctx.wavefunction(), general.wavefunction()):
        assert np.array_equal(x, y)


def test_a_wait_that_ran_out_ends_with_its_call(torch_cuda):
    # A whole-GPU launch of the last call gave up; a batch over the same context, with a
    # cut that a cluster holds, runs resident (the persistent launches would size its
    # table at three times N_MAX).
    from paper_2301_05726_gb300.api import batch_run
    p = synth.make_problem(77, 12, 4, 4, 0.08).prefix(120)
    ctx = context(p, batch_wait_ms=50, batch_test_skip_block=2)
    ctx.apply()
    assert ctx.stats()["forward_launches"] > p.n_exc
    cut = dict(n_max=2000, n_cut=1000)
    ctx.set_options(batch_wait_ms=0, batch_test_skip_block=0, **cut)
    E, grads = batch_run([ctx], 0.0)
    assert ctx.stats()["capacity_entries"] != 3 * cut["n_max"]
    assert_gradient((E[0], grads[0]), p, **cut)


def test_dropped_entries_near_the_room(torch_cuda):
    # 714,208 determinants, near the 760,000 that the GPU holds, then factors of angle
    # pi/2: each moves some 5 % of them, so that what it leaves behind is dropped.
    base = synth.make_problem(77, 24, 3, 3, 0.15, eps=1e-12)
    p = dataclasses.replace(base.prefix(260), n_max=715_000, n_cut=705_000)
    ctx = context(p)
    ctx.apply()
    keys = ctx.wavefunction()[0][::7]

    def linked(row):
        i, j, a, b = (int(x) for x in row)
        occ, vir = np.uint64((1 << i) | (1 << j)), np.uint64((1 << a) | (1 << b))
        x = keys & (occ | vir)
        return float(np.mean((x == occ) | (x == vir)))

    rows = [r for r in base.exc[260:] if r[1] >= 0]
    rows = np.array([r for r in rows if 0.045 < linked(r) < 0.06][:40], dtype=np.int32)
    assert len(rows) == 40
    p = dataclasses.replace(p, exc=np.concatenate([p.exc, rows]),
                            theta=np.concatenate([p.theta, np.full(len(rows), np.pi / 2)]))
    ctx, general = context(p), context(p, rebuild_test_regions=1)
    for c in (ctx, general):
        c.apply()
    st, sg = ctx.stats(), general.stats()
    for x in ("n_det", "rotations", "created", "dropped_new", "dropped_old", "cut"):
        assert st[x] == sg[x], x
    assert st["dropped_old"] > 500_000 and st["forward_launches"] == 1
    for x, y in zip(ctx.wavefunction(), general.wavefunction()):
        assert np.array_equal(x, y)
    ctx.gradient()  # (more tape may be needed on the way: a second launch)
    E, g = ctx.gradient()
    assert_gradient((E, g), p)
    assert ctx.stats()["forward_launches"] == 1 and ctx.stats()["reverse_launches"] == 1


@pytest.mark.parametrize("stride", [0, 15])
def test_no_reverse_pass_over_tables_that_do_not_fit(torch_cuda, stride):
    # The final state fits the GPU, a table on the way does not: the reverse sweep of the
    # factors around it takes a launch each, without a resident one before them.
    p = dataclasses.replace(doubling(20, extra=[(0, 1, 20, 21), (2, 3, 22, 23)]), n_max=1_000_000, n_cut=100_000)
    ctx = context(p, checkpoint_stride=stride)
    assert_gradient(ctx.gradient(), p, checkpoint_stride=stride)
    # (with segments the first fifteen factors run resident: one launch)
    assert ctx.stats()["reverse_launches"] == (p.n_exc if stride == 0 else p.n_exc - 15 + 1)


def test_the_first_table_of_a_small_problem(torch_cuda):
    # 36 determinants in the sector: the table has the size of any first one.
    p = synth.make_problem(77, 4, 2, 2, 0.08)
    ctx = context(p)
    ctx.apply()
    assert ctx.stats()["n_det"] <= 36 and ctx.stats()["capacity_entries"] == 4096
