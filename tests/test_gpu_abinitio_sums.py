"""The ab initio local energy where a short cut would show: more electrons than a warp
has lanes, samples that no walker wrote.
"""
import numpy as np
import pytest

import oracle
from paper_1108_0900_gb300 import inputs
from paper_1108_0900_gb300 import vmcsr as V
from test_gpu_abinitio_energy import condition, energies, problem

pytest.importorskip("torch")
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
