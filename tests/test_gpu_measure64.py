"""FP64 evaluation of given configurations at the edges of its layout: the smallest
and largest electron counts, one spin only, pairing that is zero between like spins
(every pivot has to be searched for), sites without bonds and repeated bonds.

The pairing block is compared with numpy's inverse, ln|Psi| with its determinant, E_L
with the oracle, each to 1e-12 kappa(A_occ): about 10^4 unit roundoffs times the
condition number, as elsewhere for quantities taken from an inverse.
"""
import numpy as np
import pytest

import oracle
from paper_1108_0900_gb300 import inputs
from paper_1108_0900_gb300 import vmcsr as V

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lx,ly,nu,nd,corr,singlet,n", [
    (2, 1, 1, 1, "none", False, 3), (3, 2, 4, 0, "pair", False, 9), (2, 2, 2, 2, "2x2", True, 7),
    (5, 5, 9, 9, "pair", True, 6), (6, 6, 17, 15, "2x2", False, 5), (8, 8, 32, 32, "pair", False, 2),
    (8, 8, 31, 3, "2x2", False, 5)])
def test_inverse_energy_and_amplitude(lx, ly, nu, nd, corr, singlet, n):
    wl = inputs.hubbard("m", lx, ly, nu, nd, corr, seed=2, n_walkers=1)
    M, ns = wl.M, wl.n_sites
    iu = np.triu_indices(M, 1)
    if singlet:
        wl.f = wl.f * ((iu[0] < ns) & (iu[1] >= ns))
    F = np.zeros((M, M))
    F[iu] = wl.f
    F -= F.T
    cfgs = inputs.draw_configs(np.random.default_rng(4), n, ns, nu, nd)
    A = [F[np.ix_(o, o)] for o in cfgs.astype(np.int64)]
    kappa = np.array([np.linalg.cond(a) for a in A])
    h = V.vmc_create(wl, n_walkers=n, samples_per_walker=1, walker_precision=V.VMC_FP64, keep_fp64_store=True)
    V.vmc_set_params(h, wl.C, wl.f)
    V.vmc_measure(h, cfgs)
    occ, E, cs, pf = V.vmc_get_samples(h)
    assert np.array_equal(occ, cfgs)
    pairs = [(a, b) for a in range(nu) for b in range(a + 1, nu)] + [(a, b) for a in range(nu, nu + nd) for b in range(a + 1, nu + nd)]
    pairs += [(a, b) for a in range(nu) for b in range(nu, nu + nd)]
    for s in range(n):
        X = np.linalg.inv(A[s])
        ref = np.array([X[b, a] for a, b in pairs])
        assert np.linalg.norm(pf[s] - ref) <= 1e-12 * kappa[s] * np.linalg.norm(ref)
    E_or = oracle.Problem(wl).measure(cfgs)[0]
    assert np.all(np.abs(E - E_or) <= 1e-12 * kappa * np.maximum(1.0, np.abs(E_or)))
    lnpsi = V.vmc_logpsi(h).cpu().numpy()
    k = wl.corr_param_off + cs.astype(np.int64)
    ref = np.array([0.5 * np.linalg.slogdet(a)[1] for a in A]) + np.log(np.abs(wl.C[k])).sum(1)
    assert np.all(np.abs(lnpsi - ref) <= 1e-12 * kappa)
    w = np.random.default_rng(5).standard_normal(n)
    grad = V.vmc_logpsi_backward(h, torch.from_numpy(w).cuda()).cpu().numpy()
    ref, size = np.zeros(wl.n_params), np.zeros(wl.n_params)
    p, q = (cfgs[:, [x[i] for x in pairs]].astype(np.int64) for i in (0, 1))
    idx = np.concatenate([k, wl.n_corr_params + p * M - p * (p + 1) // 2 + q - p - 1], 1)
    val = np.concatenate([1.0 / wl.C[k], pf], 1) * w[:, None]
    np.add.at(ref, idx, val)
    np.add.at(size, idx, np.abs(val))
    assert np.all(np.abs(grad - ref) <= 1e-12 * kappa.max() * size)
    h.close()


def test_singular_block_is_reported():
    wl = inputs.hubbard("m", 3, 2, 2, 2, "none", seed=2, n_walkers=1)
    wl.f = wl.f * 0.0
    h = V.vmc_create(wl, n_walkers=2, samples_per_walker=1, walker_precision=V.VMC_FP64, keep_fp64_store=True)
    V.vmc_set_params(h, wl.C, wl.f)
    with pytest.raises(V.VmcError) as err:
        V.vmc_measure(h, inputs.draw_configs(np.random.default_rng(4), 2, 6, 2, 2))
    assert err.value.code == -3
    h.close()
