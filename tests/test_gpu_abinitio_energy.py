"""The ab initio local energy's pass at the edges of its layouts: one and two
sites per lane, more than 32 electrons, empty spins and classes, sites with no,
one or several correlators, and the general correlator path.

Tolerances: E_L sums up to 10^5 excitation terms whose ratios carry the rounding
of the occupied block's inverse, so an FP64 energy is held to 1e-12 kappa(A_occ)
relative to the largest of |E_L| and 1, and an FP32 one (unit roundoff 2^29
larger) to 1e-4 kappa.
"""
import numpy as np
import pytest

import oracle
from paper_1108_0900_gb300 import inputs
from paper_1108_0900_gb300 import vmcsr as V

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def problem(n, nu, nd, corr, n_chol=3, seed=31):
    wl = inputs.abinitio("e", n, nu, nd, n_chol=n_chol, seed=seed, n_walkers=1)
    pairs = inputs.all_pair_correlators(n)
    sites = {"pairs": pairs, "none": [], "mixed": pairs[::2] + pairs[:3] + [np.asarray([i], np.int32) for i in range(0, n, 2)],
             "triples": pairs[::3] + [np.asarray([0, 1, n - 1], np.int32)]}[corr]
    wl.corr_sites = sites
    rng = np.random.default_rng(seed + 1)
    wl.C = 1.0 + 0.2 * rng.standard_normal(sum(4 ** len(s) for s in sites))
    wl.C = np.where(np.abs(wl.C) < 0.2, 0.2, wl.C)
    return wl


def energies(wl, cfgs, prec, keep64=True, keeplow=False):
    h = V.vmc_create(wl, n_walkers=len(cfgs), samples_per_walker=1, walker_precision=prec, keep_fp64_store=keep64,
                     keep_lowp_store=keeplow)
    V.vmc_set_params(h, wl.C, wl.f)
    V.vmc_measure(h, cfgs)
    _, E, _, _ = V.vmc_get_samples(h, V.VMC_STORE_FP64 if keep64 else V.VMC_STORE_FP32)
    h.close()
    return E


def condition(wl, cfgs):
    M = wl.M
    F = np.zeros((M, M))
    F[np.triu_indices(M, 1)] = wl.f
    F -= F.T
    return np.array([np.linalg.cond(F[np.ix_(o, o)]) for o in cfgs.astype(np.int64)])


@pytest.mark.parametrize("n,nu,nd,corr,count", [
    (5, 1, 3, "pairs", 40), (6, 3, 3, "mixed", 40), (9, 4, 2, "none", 20), (7, 0, 4, "pairs", 20), (4, 4, 2, "pairs", 6),
    (8, 3, 3, "triples", 20), (14, 7, 7, "pairs", 6), (33, 2, 2, "pairs", 3), (34, 18, 18, "pairs", 1)])
def test_energy_matches_oracle(n, nu, nd, corr, count):
    wl = problem(n, nu, nd, corr)
    cfgs = inputs.draw_configs(np.random.default_rng(n), count, n, nu, nd)
    E_or = oracle.Problem(wl).measure(cfgs)[0]
    kappa, scale = condition(wl, cfgs), np.maximum(1.0, np.abs(E_or))
    assert np.all(np.abs(energies(wl, cfgs, V.VMC_FP64) - E_or) <= 1e-12 * kappa * scale)
    # FP64 walkers that keep the 32-bit stores only: the same pass over a block of its own
    assert np.array_equal(energies(wl, cfgs, V.VMC_FP64, False, True), energies(wl, cfgs, V.VMC_FP64))
    E32 = energies(wl, cfgs, V.VMC_FP32, False, True)
    assert np.all(np.abs(E32 - E_or) <= 1e-4 * kappa * scale)
    # the stored 32-bit block is exact in either store
    assert np.array_equal(energies(wl, cfgs, V.VMC_FP32), E32)


@pytest.mark.parametrize("symmetric", [True, False])
def test_tables_equal_the_general_correlator_path(symmetric):
    """A correlator over three sites with all amplitudes one changes nothing but sends the
    energy down the general path: equal energies, also for factors L^mu that are not
    symmetric (whose integrals are not packed)."""
    wl = problem(12, 6, 4, "mixed")
    if not symmetric:
        wl.chol = wl.chol + 0.1 * np.random.default_rng(3).standard_normal(wl.chol.shape)
    cfgs = inputs.draw_configs(np.random.default_rng(2), 50, 12, 6, 4)
    E = energies(wl, cfgs, V.VMC_FP64)
    wl.corr_sites = wl.corr_sites + [np.asarray([2, 5, 7], np.int32)]
    wl.C = np.concatenate([wl.C, np.ones(64)])
    ref = energies(wl, cfgs, V.VMC_FP64)
    assert np.all(np.abs(E - ref) <= 1e-12 * condition(wl, cfgs) * np.maximum(1.0, np.abs(ref)))
