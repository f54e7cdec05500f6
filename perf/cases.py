"""The work this framework is used for, as cases that a measurement can run.

A case is one problem shape and one kind of call through the public Python face of the library
(``UCCContext``, ``ucc_energy``, ``batch_run``).  A pass hands over a vector of angles, as every step of an
optimiser or a scan does, and takes back what the call computes.  The kinds:

* ``gradient``  E and dE/dtheta of every factor: one step of the variational optimisation;
* ``autograd``  the same through the torch op, with the angles on the device;
* ``energy``    E and <psi|psi>: a line search, a finite difference, fixed angles at another cut;
* ``entropy``   the Eq. 6 entropy after every factor, and E;
* ``state``     the determinants, their amplitudes and sigma = P_S H psi, read back to the host, and E;
* ``batch``     E and gradients of many independent problems in one call.

Problems are the seeded synthetic ones of ``synth`` in the shapes that its workloads, the tests and the
benchmark use: ``md`` doubles of largest |theta| (0: all) and all singles, eps, and the N_MAX/N_CUT cut.
"""
import functools
import math

import numpy as np
import torch

from paper_2301_05726_gb300 import synth
from paper_2301_05726_gb300.api import UCCContext, batch_run, ucc_energy


def _case(name, kind, n_spatial, n_alpha, n_beta, sigma, eps=0.0, md=0, n_max=0, n_cut=0, stride=0, jobs=0):
    c = dict(kind=kind, n_spatial=n_spatial, n_alpha=n_alpha, n_beta=n_beta, sigma=sigma, eps=eps, md=md,
             n_max=n_max, n_cut=n_cut, stride=stride, jobs=jobs)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # A small molecule in a minimal basis, optimised to convergence: 92 factors, 225 determinants.
        _case("gradient_12so", "gradient", 6, 2, 2, 0.05),
        # The entropy curve of a 16-qubit, 10-electron molecule: 315 factors, 3,136 determinants.
        _case("entropy_16so", "entropy", 8, 5, 5, 0.05),
        # The exact 24-spin-orbital state: one energy, as a line search or a finite difference asks for it.
        _case("energy_24so", "energy", 12, 4, 4, 0.02),
        # One optimisation step of the same problem from a torch program: 1,424 factors, 245,025 determinants.
        _case("autograd_24so", "autograd", 12, 4, 4, 0.02),
        # An open-shell doublet, its state read back with sigma, as a selected-CI step wants it.
        _case("state_30so", "state", 15, 4, 3, 0.02),
        # The production setting of the 64-qubit study (M_D = 5,000, N_MAX = 8,000, N_CUT = 5,000): one step.
        _case("gradient_64so_cut8000", "gradient", 32, 5, 5, 0.02, md=5000, n_max=8000, n_cut=5000),
        # The same study's fixed angles with the state allowed to grow.
        _case("energy_64so_cut160000", "energy", 32, 5, 5, 0.02, md=5000, n_max=160000, n_cut=100000),
        # A frozen-core 72-spin-orbital problem: two-word keys, the production cut.
        _case("gradient_72so_cut8000", "gradient", 36, 6, 6, 0.02, eps=1e-8, md=5000, n_max=8000, n_cut=5000),
        # A scan of 24 uneven molecules (16-36 spin-orbitals, 4-12 electrons) in one call.
        _case("batch_24_jobs", "batch", 0, 0, 0, 0.02, eps=1e-8, n_max=8000, n_cut=5000, jobs=24),
        # 40 spin-orbitals up to 1e7 determinants, gradient with sqrt(K) checkpoints.
        _case("gradient_40so_ckpt", "gradient", 20, 6, 6, 0.01, eps=1e-8, md=400, n_max=10_000_000,
              n_cut=6_250_000, stride=26),
        # 64 spin-orbitals up to 1e7 determinants: the benchmark's problem with fewer doubles.
        _case("gradient_64so_cut1e7", "gradient", 32, 8, 8, 0.005, eps=1e-6, md=1800, n_max=10_000_000,
              n_cut=6_250_000),
    ]


def _n_singles(n, a, b):
    return a * (n - a) + b * (n - b)


def _n_doubles(n, a, b):
    return (math.comb(a, 2) * math.comb(n - a, 2) + math.comb(b, 2) * math.comb(n - b, 2)
            + a * b * (n - a) * (n - b))


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: small and exact, mid-sized and exact, the production cut, a
    larger cut, a map near 1e7, two-word keys, or a batch."""
    family = rng.choice(["small", "mid", "cut", "cut", "grown", "large", "wide", "batch"])
    if family == "small":
        n = rng.randint(4, 9)
        a, b = rng.randint(1, n // 2 + 1), rng.randint(1, n // 2 + 1)
        kind = rng.choice(["gradient", "energy", "entropy", "state", "autograd"])
        # a state that is read back is whole: how many determinants eps leaves would depend on the angles
        return _case("", kind, n, a, b, 0.05, eps=0.0 if kind == "state" else rng.choice([0.0, 1e-8, 1e-5]))
    if family == "mid":
        n = rng.randint(10, 13)
        a, b = rng.randint(2, 4), rng.randint(2, 4)
        kind = rng.choice(["gradient", "energy", "state", "autograd"])
        if kind == "state":
            return _case("", kind, n, a, b, 0.02)
        return _case("", kind, n, a, b, 0.02, eps=rng.choice([0.0, 0.0, 1e-8]), md=_log(rng, 100, 1000))
    if family == "cut":
        n, a = rng.randint(16, 32), rng.randint(3, 7)
        n_cut = _log(rng, 1000, 10000)
        return _case("", rng.choice(["gradient", "energy"]), n, a, max(3, a - rng.randint(0, 1)), 0.02,
                     eps=rng.choice([0.0, 1e-8]), md=_log(rng, 300, 4500), n_max=8 * n_cut // 5, n_cut=n_cut)
    if family == "grown":
        n, a = rng.randint(18, 32), rng.randint(4, 6)
        n_cut = _log(rng, 10000, 500000)
        return _case("", rng.choice(["gradient", "energy"]), n, a, a, 0.02, eps=rng.choice([0.0, 1e-8]),
                     md=_log(rng, 200, 1500), n_max=8 * n_cut // 5, n_cut=n_cut)
    if family == "large":
        n, a = rng.randint(20, 32), rng.randint(6, 8)
        n_cut = _log(rng, 500000, 6000000)
        return _case("", "gradient", n, a, a, 0.005, eps=1e-6, md=_log(rng, 200, 1200), n_max=8 * n_cut // 5,
                     n_cut=n_cut, stride=rng.choice([0, 0, 40]))
    if family == "wide":
        n, a = rng.randint(33, 40), rng.randint(4, 6)
        n_cut = _log(rng, 1000, 20000)
        return _case("", rng.choice(["gradient", "energy"]), n, a, a, 0.02, eps=1e-8, md=_log(rng, 300, 4000),
                     n_max=8 * n_cut // 5, n_cut=n_cut)
    n_cut = _log(rng, 1000, 5000)
    return _case("", "batch", 0, 0, 0, 0.02, eps=1e-8, n_max=8 * n_cut // 5, n_cut=n_cut, jobs=rng.randint(2, 20))


@functools.lru_cache(maxsize=None)
def _excitations(n, a, b):
    return synth.enumerate_excitations(n, a, b)


def _problem(case, seed, n=None, a=None, b=None):
    n, a, b = (case["n_spatial"], case["n_alpha"], case["n_beta"]) if n is None else (n, a, b)
    rng = np.random.default_rng(seed)
    h, g = synth.make_integrals(rng, n)
    s, d = _excitations(n, a, b)
    th_s = rng.normal(0.0, case["sigma"], size=len(s))
    th_d = rng.normal(0.0, case["sigma"], size=len(d))
    exc, theta = synth.order_and_truncate(s, d, th_s, th_d, case["md"] or None)
    return synth.Problem(n, a, b, h, g, exc, theta, eps=case["eps"], n_max=case["n_max"], n_cut=case["n_cut"])


def _problems(case, seed):
    if case["kind"] != "batch":
        return [_problem(case, seed)]
    shapes = [synth.batch_job_shape(j) for j in range(case["jobs"])]
    return [_problem(case, 1000 * seed + j, *shape) for j, shape in enumerate(shapes)]


def prepare(case, seed):
    ctxs = []
    for p in _problems(case, seed):
        c = UCCContext(p)
        if case["stride"]:
            c.set_options(checkpoint_stride=case["stride"])
        if case["kind"] == "entropy":
            c.set_options(record_entropy=1)
        ctxs.append(c)
    theta = [c.prob.theta.copy() for c in ctxs]
    if case["kind"] == "autograd":
        theta = [torch.tensor(t, dtype=torch.float64, device="cuda", requires_grad=True) for t in theta]
    return dict(kind=case["kind"], eps=case["eps"], ctxs=ctxs, theta=theta)


def run(state):
    kind, ctxs = state["kind"], state["ctxs"]
    if kind == "autograd":
        E = ucc_energy(ctxs[0], state["theta"][0])
        (grad,) = torch.autograd.grad(E, state["theta"][0])
        return dict(E=E.detach(), grad=grad)
    for c, t in zip(ctxs, state["theta"]):
        c.set_theta(t)
    if kind == "batch":
        E, grads = batch_run(ctxs, state["eps"], with_grad=True)
        return dict(E=E, grads=grads)
    ctx = ctxs[0]
    if kind == "gradient":
        E, grad = ctx.gradient()
        return dict(E=E, grad=grad)
    ctx.apply()
    E, norm2 = ctx.energy()
    if kind == "energy":
        return dict(E=E, norm2=norm2)
    if kind == "entropy":
        return dict(E=E, norm2=norm2, entropy=ctx.entropy())
    keys, amps, sigma = ctx.wavefunction(with_sigma=True)
    return dict(E=E, norm2=norm2, keys=keys.view(np.int64), amps=amps, sigma=sigma)


def _shape(case):
    """(spatial orbitals, factors, stored determinants at most) of every problem of a case."""
    shapes = ([synth.batch_job_shape(j) for j in range(case["jobs"])] if case["kind"] == "batch"
              else [(case["n_spatial"], case["n_alpha"], case["n_beta"])])
    for n, a, b in shapes:
        d = _n_doubles(n, a, b)
        sector = synth.hilbert_size(n, a, b)
        yield n, (min(case["md"], d) if case["md"] else d) + _n_singles(n, a, b), \
            min(sector, case["n_max"]) if case["n_max"] else sector


def work(case):
    """Inputs (integrals, factor rows, angles) read once and results written once; the arithmetic of the
    rotations of a state that is at its full size half of the time, a quarter of it linked by a factor:
    six operations a pair forward, and thirteen more where the gradient goes back over it."""
    grad = case["kind"] in ("gradient", "autograd", "batch")
    bytes_ = flops = 0
    for n, k, d in _shape(case):
        bytes_ += 8 * (n * n + n ** 4) + 24 * k + 16
        bytes_ += 8 * k if grad or case["kind"] == "entropy" else 0
        bytes_ += 24 * d if case["kind"] == "state" else 0
        flops += k * d / 8 * (19 if grad else 6)
    return dict(bytes=bytes_, flops=flops)


# ---------------------------------------------------------------------------
# The same results from plain torch operations in 64 bits: the state as sorted keys and amplitudes, one
# factor at a time by its definition; E from every single and double excitation of every determinant;
# the gradient from the kept states of every factor.
# ---------------------------------------------------------------------------
def _i64(x):
    return x - (1 << 64) if x >= (1 << 63) else x


def _parity(x):
    for s in (32, 16, 8, 4, 2, 1):
        x = x ^ (x >> s)
    return x & 1


def _sign(keys, ops):
    """Sign of the product of ladder operators on orbitals ops, applied in that order to keys that they do
    not annihilate; an operator counts the occupied modes below its orbital."""
    par = torch.zeros_like(keys)
    for p in ops:
        par = par ^ _parity(keys & _i64((1 << p) - 1))
        keys = keys ^ _i64(1 << p)
    return 1.0 - 2.0 * par.double()


def _find(keys, query):
    at = torch.searchsorted(keys, query).clamp_(max=keys.numel() - 1)
    return at, keys[at] == query


def _take(keys, vals, query):
    at, hit = _find(keys, query)
    return torch.where(hit, vals[at], 0.0)


class _Factor:
    def __init__(self, row, theta):
        i, j, a, b = (int(x) for x in row)
        occ, vir = (i,) if j < 0 else (i, j), (a,) if j < 0 else (a, b)
        self.ops = (i, a) if j < 0 else (i, j, b, a)
        self.occ, self.vir = (_i64(sum(1 << p for p in m)) for m in (occ, vir))
        self.m = self.occ | self.vir
        self.c, self.s = math.cos(theta), math.sin(theta)

    def pairs(self, keys):
        """The members E and D of every pair with a stored one, and the sign of tau|E> = s|D>."""
        on = keys & self.m
        e, d = keys[on == self.occ], keys[on == self.vir] ^ self.m
        if e.numel():
            d = d[~_find(e, d)[1]]
        e = torch.cat([e, d])
        return e, e ^ self.m, _sign(e, self.ops)


def _cut(keys, amps, n_max, n_cut):
    if not n_max or keys.numel() <= n_max:
        return keys, amps
    unsigned = torch.sort(keys ^ _i64(1 << 63)).indices  # ties go to the smaller key
    keep = unsigned[torch.sort(-amps[unsigned].abs(), stable=True).indices[:n_cut]].sort().values
    return keys[keep], amps[keep]


def _forward(p, factors, keep_all):
    keys = torch.tensor([_i64(p.hf_key)], device="cuda")
    amps = torch.ones(1, dtype=torch.float64, device="cuda")
    states, entropy = [(keys, amps)], []
    for f in factors:
        e, d, s = f.pairs(keys)
        ss = s * f.s
        cE, cD = _take(keys, amps, e), _take(keys, amps, d)
        nE, nD = f.c * cE - ss * cD, f.c * cD + ss * cE
        rest = (keys & f.m)
        rest = (rest != f.occ) & (rest != f.vir)
        n, c = torch.cat([e, d]), torch.cat([nE, nD])
        kept = c.abs() >= p.eps
        keys, order = torch.sort(torch.cat([keys[rest], n[kept]]))
        amps = torch.cat([amps[rest], c[kept]])[order]
        keys, amps = _cut(keys, amps, p.n_max, p.n_cut)
        if keep_all:
            states.append((keys, amps))
        else:
            w = amps * amps
            entropy.append(-(torch.xlogy(w, w)).sum())
    return keys, amps, states, entropy


def _sigma(p, keys, amps):
    """P_S H psi: every connection of a chunk of determinants, those that are stored kept."""
    n, n_so = p.n_spatial, p.n_so
    h, g = torch.tensor(p.h, device="cuda"), torch.tensor(p.g, device="cuda")
    bit = torch.tensor([_i64(1 << q) for q in range(n_so)], device="cuda")
    sig = torch.zeros_like(amps)
    conn = _n_doubles(n, p.n_alpha, p.n_beta) + 1
    for at in range(0, keys.numel(), max(1, (1 << 25) // conn)):
        I = keys[at:at + max(1, (1 << 25) // conn)]
        on = (I[:, None] & bit) != 0
        occ = [on[:, s::2].nonzero()[:, 1].view(I.numel(), -1) * 2 + s for s in (0, 1)]
        vir = [(~on[:, s::2]).nonzero()[:, 1].view(I.numel(), -1) * 2 + s for s in (0, 1)]
        every = torch.cat(occ, 1)
        oo = every // 2
        acc = h[oo, oo].sum(1)  # the diagonal
        x, y = oo[:, :, None], oo[:, None, :]
        same = (every[:, :, None] & 1) == (every[:, None, :] & 1)
        acc = (acc + 0.5 * (g[x, x, y, y] - torch.where(same, g[x, y, y, x], 0.0)).sum((1, 2))) * amps[at:at + I.numel()]

        def hits(J):
            pos, hit = _find(keys, J.reshape(-1))
            at_hit = hit.nonzero()[:, 0]
            return at_hit, amps[pos[at_hit]]

        def below(q):
            return torch.where(q >= 63, torch.full_like(q, (1 << 63) - 1), bit[q] - 1)

        def signed(K, ops):
            par = torch.zeros_like(K)
            for q in ops:
                par = par ^ _parity(K & below(q))
                K = K ^ bit[q]
            return 1.0 - 2.0 * par.double()

        for s in (0, 1):
            no, nv = occ[s].shape[1], vir[s].shape[1]
            if not no or not nv:
                continue
            J = (I[:, None, None] ^ bit[occ[s]][:, :, None]) ^ bit[vir[s]][:, None, :]
            t, c = hits(J)
            r0, o, v = t // (no * nv), (t // nv) % no, t % nv
            q, r = occ[s][r0, o], vir[s][r0, v]
            k = every[r0]
            el = h[r // 2, q // 2] + g[(r // 2)[:, None], (q // 2)[:, None], k // 2, k // 2].sum(1)
            el = el - torch.where((k & 1) == s, g[(r // 2)[:, None], k // 2, k // 2, (q // 2)[:, None]], 0.0).sum(1)
            acc.index_add_(0, r0, el * signed(I[r0], (q, r)) * c)
            if no < 2 or nv < 2:
                continue
            io, jo = torch.triu_indices(no, no, 1, device="cuda")
            iv, jv = torch.triu_indices(nv, nv, 1, device="cuda")
            J = (I[:, None] ^ bit[occ[s][:, io]] ^ bit[occ[s][:, jo]])[:, :, None] ^ \
                (bit[vir[s][:, iv]] ^ bit[vir[s][:, jv]])[:, None, :]
            t, c = hits(J)
            r0, o, v = t // (io.numel() * iv.numel()), (t // iv.numel()) % io.numel(), t % iv.numel()
            q1, q2, r1, r2 = occ[s][r0, io[o]], occ[s][r0, jo[o]], vir[s][r0, iv[v]], vir[s][r0, jv[v]]
            el = g[r1 // 2, q1 // 2, r2 // 2, q2 // 2] - g[r1 // 2, q2 // 2, r2 // 2, q1 // 2]
            acc.index_add_(0, r0, el * signed(I[r0], (q1, q2, r2, r1)) * c)
        no, mo, nv, mv = occ[0].shape[1], occ[1].shape[1], vir[0].shape[1], vir[1].shape[1]
        if no and mo and nv and mv:
            J = (I[:, None, None] ^ bit[occ[0]][:, :, None] ^ bit[occ[1]][:, None, :]).view(I.numel(), -1)[:, :, None] ^ \
                (bit[vir[0]][:, :, None] ^ bit[vir[1]][:, None, :]).view(I.numel(), -1)[:, None, :]
            t, c = hits(J)
            r0, o, v = t // (no * mo * nv * mv), (t // (nv * mv)) % (no * mo), t % (nv * mv)
            q1, q2, r1, r2 = occ[0][r0, o // mo], occ[1][r0, o % mo], vir[0][r0, v // mv], vir[1][r0, v % mv]
            el = g[r1 // 2, q1 // 2, r2 // 2, q2 // 2]
            acc.index_add_(0, r0, el * signed(I[r0], (q1, q2, r2, r1)) * c)
        sig[at:at + I.numel()] = acc
    return sig


def _gradient(factors, states, sig, E, norm2):
    lam = (sig - E * states[-1][1]) / norm2
    grad = torch.zeros(len(factors), dtype=torch.float64, device="cuda")
    for k in range(len(factors) - 1, -1, -1):
        f, after = factors[k], states[k + 1][0]
        keys, amps = states[k]
        e, d, s = f.pairs(keys)
        ss = s * f.s
        muE, muD = _take(after, lam, e), _take(after, lam, d)
        lE, lD = f.c * muE + ss * muD, f.c * muD - ss * muE
        grad[k] = 2.0 * (s * (lD * _take(keys, amps, e) - lE * _take(keys, amps, d))).sum()
        lam = _take(after, lam, keys)
        for who, val in ((e, lE), (d, lD)):
            at, hit = _find(keys, who)
            lam[at[hit]] = val[hit]
    return grad


def exact(case, seed):
    if case["kind"] == "batch" or case["n_spatial"] > 32 or case["n_spatial"] == 0:
        return None
    (n, k, d), = _shape(case)
    grad = case["kind"] in ("gradient", "autograd")
    connections = d * (_n_doubles(n, case["n_alpha"], case["n_beta"]) + _n_singles(n, case["n_alpha"], case["n_beta"]))
    if connections > 1e9 or k * (0.0015 + 2e-8 * d) * (2 if grad else 1) > 20 or k * d * 16 > 2e10:
        return None
    p = _problem(case, seed)
    factors = [_Factor(row, t) for row, t in zip(p.exc, p.theta)]
    keys, amps, states, entropy = _forward(p, factors, grad)
    sig = _sigma(p, keys, amps)
    norm2 = float((amps * amps).sum())
    E = float((amps * sig).sum()) / norm2 + p.e_nuc
    if case["kind"] == "autograd":
        E64 = torch.tensor(E, dtype=torch.float64)
        return dict(E=E64, grad=_gradient(factors, states, sig, E, norm2))
    if grad:
        return dict(E=E, grad=_gradient(factors, states, sig, E, norm2))
    if case["kind"] == "energy":
        return dict(E=E, norm2=norm2)
    if case["kind"] == "entropy":
        return dict(E=E, norm2=norm2, entropy=torch.stack(entropy))
    order = torch.sort(keys ^ _i64(1 << 63)).indices
    return dict(E=E, norm2=norm2, keys=None, amps=amps[order], sigma=sig[order])
