"""The ab initio local energy where a short cut would show: more electrons than a warp
has lanes, samples that no walker wrote, sample sets larger than the workspace,
sums that FP32 cannot hold, integrals of zero beside ratios that overflow,
correlators whose single toggles leave the walker's range.
"""
import itertools

import numpy as np
import pytest

import oracle
from paper_1108_0900_gb300 import inputs
from paper_1108_0900_gb300 import vmcsr as V
from test_gpu_abinitio_energy import condition, energies, problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nu,nd,corr,count", [
    (20, 18, 18, "pairs", 2), (24, 20, 20, "pairs", 1), (20, 17, 17, "pairs", 2), (32, 31, 31, "none", 2),
    (17, 17, 17, "triples", 1), (20, 18, 16, "triples", 1), (32, 32, 32, "pairs", 1)])
def test_more_electrons_than_lanes(n, nu, nd, corr, count):
    """More than 32 electrons in at most 32 orbitals; tolerances as in
    test_gpu_abinitio_energy.py."""
    wl = problem(n, nu, nd, corr)
    cfgs = inputs.draw_configs(np.random.default_rng(n), count, n, nu, nd)
    E_or = oracle.Problem(wl).measure(cfgs)[0]
    kappa, scale = condition(wl, cfgs), np.maximum(1.0, np.abs(E_or))
    assert np.all(np.abs(energies(wl, cfgs, V.VMC_FP64) - E_or) <= 1e-12 * kappa * scale)
    assert np.all(np.abs(energies(wl, cfgs, V.VMC_FP32, False, True) - E_or) <= 1e-4 * kappa * scale)


@pytest.mark.parametrize("prec", [V.VMC_FP32, V.VMC_FP64])
def test_samples_that_no_walker_wrote_are_passed_over(prec):
    """A pairing without partners for up orbital 0 makes every configuration that holds it
    singular: on a fresh handle nothing is written for it.  The others' energies are those of a
    set of their own."""
    n, ne = 10, 4
    wl = problem(n, ne, ne, "mixed")
    F = np.zeros((2 * n, 2 * n))
    F[np.triu_indices(2 * n, 1)] = wl.f
    F[0] = 0.0
    wl.f = F[np.triu_indices(2 * n, 1)]
    cfgs = inputs.draw_configs(np.random.default_rng(3), 60, n, ne, ne)
    bad = (cfgs == 0).any(1)
    assert 10 < bad.sum() < 50
    h = V.vmc_create(wl, n_walkers=len(cfgs), samples_per_walker=1, walker_precision=prec)
    V.vmc_set_params(h, wl.C, wl.f)
    with pytest.raises(V.VmcError, match="SINGULAR"):
        V.vmc_measure(h, cfgs[bad])
    with pytest.raises(V.VmcError, match="SINGULAR"):
        V.vmc_measure(h, cfgs)
    E = V.vmc_get_samples(h)[1]
    h.close()
    assert np.array_equal(E[~bad], energies(wl, cfgs[~bad], prec))


@pytest.mark.parametrize("refresh", [False, True])
def test_sampling_takes_no_device_memory(refresh):
    """What sampling and measuring need is there when the handle is."""
    wl = problem(12, 6, 6, "pairs")
    occ = inputs.draw_configs(np.random.default_rng(1), 2048, 12, 6, 6)

    def free_before_and_after():
        h = V.vmc_create(wl, n_walkers=2048, samples_per_walker=4, walker_precision=V.VMC_FP32, fp64_refresh=refresh)
        V.vmc_set_params(h, wl.C, wl.f)
        V.vmc_set_walkers(h, occ)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        V.vmc_sample(h, 1, 7)
        V.vmc_measure(h, occ)
        V.vmc_logpsi_backward(h)
        torch.cuda.synchronize()
        after = torch.cuda.mem_get_info()[0]
        h.close()
        return before, after

    free_before_and_after()   # loads the kernels
    before, after = free_before_and_after()
    assert after == before


def test_sample_sets_beyond_the_inverses_workspace():
    """1.1 million samples of 16 electrons in FP64 hold more inverses than the workspace: they
    go in pieces, with the samples and energies of a handle that needs one."""
    wl = problem(9, 8, 8, "pairs")
    nw, spw, few = 550001, 2, 3000
    base = inputs.draw_configs(np.random.default_rng(1), 81, 9, 8, 8)
    occ = np.ascontiguousarray(base[np.arange(nw) % len(base)])
    h = V.vmc_create(wl, n_walkers=nw, samples_per_walker=spw)
    g = V.vmc_create(wl, n_walkers=few, samples_per_walker=spw)
    for x, o in ((h, occ), (g, occ[:few])):
        V.vmc_set_params(x, wl.C, wl.f)
        V.vmc_set_walkers(x, o)
        V.vmc_sample(x, 1, 77)
    so, sE, _, _ = V.vmc_get_samples(h)
    go, gE, _, _ = V.vmc_get_samples(g)
    assert np.array_equal(so[:few * spw], go) and np.array_equal(sE[:few * spw], gE)
    # a configuration's energy does not depend on where it is evaluated
    pick = np.random.default_rng(2).integers(0, nw * spw, few * spw)
    V.vmc_measure(h, so)
    mE = V.vmc_get_samples(h)[1]
    V.vmc_measure(g, np.ascontiguousarray(so[pick]))
    assert np.array_equal(V.vmc_get_samples(g)[1], mE[pick])
    # nor on the chain, but for the drift of its rank-2 updates (1e-16 per update, times the
    # condition of the blocks on the way); another sample's energy would be off by order one
    assert np.mean(np.abs(sE[pick] - mE[pick]) <= 1e-6 * np.maximum(1.0, np.abs(mE[pick]))) >= 0.99
    h.close()
    g.close()


def singlet(n, phi, chol, h=None, corr_sites=(), C=None):
    """Pairing f between up orbital i and down orbital j = phi[i, j] only."""
    M = 2 * n
    F = np.zeros((M, M))
    F[:n, n:] = phi
    sites = [np.asarray(s, np.int32) for s in corr_sites]
    return inputs.Workload(name="s", n_sites=n, n_up=1, n_dn=1, ham=inputs.ABINITIO, corr_sites=sites,
                           C=np.zeros(0) if C is None else C, f=F[np.triu_indices(M, 1)],
                           h=np.zeros((n, n)) if h is None else h, chol=chol, n_walkers=1)


@pytest.mark.parametrize("prec", [V.VMC_FP32, V.VMC_FP64])
def test_diagonal_is_summed_beyond_fp32(prec):
    """Diagonal factors L^mu: E_L is <n|H|n> alone, (kk|ll) odd integers below 2^22 (exact
    in FP32) whose sum over pairs passes 2^24.  FP64 sums are exact."""
    n, ne = 12, 6
    rng = np.random.default_rng(5)
    l = 2.0 * rng.integers(512, 1024, n) + 1.0
    hd = rng.integers(1, 1 << 20, n).astype(np.float64)
    phi = rng.standard_normal((n, n))
    wl = singlet(n, phi, np.diag(l)[None], np.diag(hd))
    wl.n_up = wl.n_dn = ne
    cfgs = inputs.draw_configs(rng, 20, n, ne, ne)
    want = []
    for o in cfgs.astype(np.int64):
        s = o % n
        w = np.outer(l[s], l[s])   # (kk|ll); the exchange (kl|lk), k != l of one spin, vanishes
        same = (o[:, None] >= n) == (o[None, :] >= n)
        w[same & (s[:, None] == s[None, :])] = 0.0
        want.append(hd[s].sum() + 0.5 * w.sum())
    want = np.array(want)
    assert want.max() > 2.0 ** 24
    assert np.array_equal(energies(wl, cfgs, prec, prec == V.VMC_FP64, prec == V.VMC_FP32), want)


@pytest.mark.parametrize("prec", [V.VMC_FP32, V.VMC_FP64])
def test_every_double_excitation_enters_the_wide_sum(prec):
    """Factors between occupied and empty orbitals only: E_L is the double excitations
    alone.  Integrals (small odd numbers times powers of two, one of the two of a
    same-spin move zero or both equal) and amplitude ratios (integers, by an identity
    pairing of the occupied block) make every term exact in FP32; a sum in FP32
    rounds, one in FP32 pairs keeps 48 bits."""
    n, ne = 26, 6
    rng = np.random.default_rng(11)
    O, X = np.arange(ne), np.arange(ne, n)
    phi = rng.integers(-1, 2, (n, n))
    phi[np.ix_(O, O)] = np.eye(ne)
    u = (2 * rng.integers(0, 4, n) + 1) * 2 ** np.where(np.arange(n) < ne, 0, rng.choice([0, 14], n)) * rng.choice([-1, 1], n)
    L = np.zeros((1, n, n))
    L[0][:3, 6:16] = np.outer(u[:3], u[6:16])
    L[0][3:6, 16:] = np.outer(u[3:6], u[16:])
    L[0] += L[0].T
    wl = singlet(n, phi.astype(np.float64), L)
    wl.n_up = wl.n_dn = ne
    cfg = np.concatenate([O, O + n]).astype(np.uint8)[None]
    Li = L[0].astype(np.int64)

    def ratio(rows, cols):
        return int(np.rint(np.linalg.det(phi[np.ix_(rows, cols)].astype(np.float64))))

    terms = []
    for a, x in itertools.product(O, X):          # up a -> x, down b -> y
        rows = np.where(O == a, x, O)
        terms += [int(Li[a, x] * Li[b, y]) * ratio(rows, np.where(O == b, y, O)) for b, y in itertools.product(O, X)]
    for a, b in itertools.combinations(O, 2):     # two of one spin
        for x, y in itertools.combinations(X, 2):
            to = np.where(O == a, x, np.where(O == b, y, O))
            m = int(Li[a, x] * Li[b, y] - Li[a, y] * Li[b, x])
            terms += [m * ratio(to, O), m * ratio(O, to)]
    assert all(t == int(np.float32(t)) for t in terms)
    E = energies(wl, cfg, prec, prec == V.VMC_FP64, prec == V.VMC_FP32)
    # about 100 additions per lane, each good to 2^-48 of the lane's sum of magnitudes
    assert abs(E[0] - sum(terms)) <= 2.0 ** -40 * sum(map(abs, terms))


@pytest.mark.parametrize("prec,big", [(V.VMC_FP32, 1e25), (V.VMC_FP64, 1e200)])
def test_vanishing_integrals_meet_no_ratio(prec, big):
    """Pairing amplitudes of the empty orbitals so large that the ratios of double moves
    overflow: with integrals of zero these moves do not enter E_L."""
    n, ne = 8, 4
    rng = np.random.default_rng(9)
    O, X = np.arange(ne), np.arange(ne, n)
    phi = rng.standard_normal((n, n))
    phi[X] *= big
    phi[np.ix_(O, X)] *= big
    hd = rng.integers(1, 100, n).astype(np.float64)
    l = 1.0 + np.arange(n)
    wl = singlet(n, phi, np.diag(l)[None], np.diag(hd))
    wl.n_up = wl.n_dn = ne
    cfg = np.concatenate([O, O + n]).astype(np.uint8)[None]
    w = np.outer(l[O], l[O])
    want = 2.0 * hd[O].sum() + 0.5 * (4.0 * w.sum() - 2.0 * np.trace(w))   # no self interaction
    assert energies(wl, cfg, prec, prec == V.VMC_FP64, prec == V.VMC_FP32)[0] == want


@pytest.mark.parametrize("prec,single", [(V.VMC_FP32, 1e-6), (V.VMC_FP32, 1e6), (V.VMC_FP64, 1e-40)])
def test_correlators_that_project_single_occupancy(prec, single):
    """Pair correlators that suppress (or favour) singly occupied sites by `single` each:
    the 13 factors of one site together leave the precision's range, those of moving
    a pair of electrons stay near one.  Tolerances as in test_gpu_abinitio_energy.py."""
    n, ne = 14, 7
    wl = problem(n, ne, ne, "pairs")
    rng = np.random.default_rng(17)
    u = np.array([1.0, single, single, 1.0]) if single < 1.0 else np.array([1.0 / single, 1.0, 1.0, 1.0 / single])
    C = np.concatenate([np.outer(u, u).reshape(-1) for _ in wl.corr_sites])
    wl.C = C * (1.0 + 0.05 * rng.uniform(-1.0, 1.0, len(C)))
    up = inputs.draw_configs(rng, 4, n, ne, ne)[:, :ne]
    if single < 1.0:
        cfgs = np.concatenate([up, up + n], 1).astype(np.uint8)     # closed shells
    else:
        empty = np.array([[s for s in range(n) if s not in set(r)] for r in up])
        cfgs = np.concatenate([up, empty + n], 1).astype(np.uint8)  # every site singly occupied
    E_or = oracle.Problem(wl).measure(cfgs)[0]
    assert np.all(np.isfinite(E_or))
    kappa, scale = condition(wl, cfgs), np.maximum(1.0, np.abs(E_or))
    eps = 1e-4 if prec == V.VMC_FP32 else 1e-12
    E = energies(wl, cfgs, prec, prec == V.VMC_FP64, prec == V.VMC_FP32)
    assert np.all(np.abs(E - E_or) <= eps * kappa * scale)
