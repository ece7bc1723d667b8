"""Linear-method products on the correlator forms that take different paths: one
and two sites, repeated pairs, more correlators on a site than the shared
table's masks hold, triples next to pairs, none, one spin only, and lattices
where few moves are reached by a factor.  Tolerances of test_gpu_lm.py: FP64
store 1e-10, FP32 store 2e-4 (relative 2-norm).
"""
import numpy as np
import pytest

import oracle
from paper_1108_0900_gb300 import inputs
from paper_1108_0900_gb300 import vmcsr as V

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def correlators(kind, n):
    pairs = inputs.all_pair_correlators(n)
    ones = [np.asarray([i], np.int32) for i in range(n)]
    return {"mixed": pairs + pairs[:4] + [p[::-1].copy() for p in pairs[::3]] + ones[::2], "none": [],
            "many": pairs * 14, "triples": pairs[::2] + [np.asarray([0, n - 1, 1], np.int32)] + ones[:2]}[kind]


@pytest.mark.parametrize("ham,n,nu,nd,kind", [
    ("abinitio", 6, 3, 3, "mixed"), ("abinitio", 6, 2, 4, "many"), ("abinitio", 5, 3, 1, "triples"),
    ("abinitio", 5, 0, 2, "mixed"), ("abinitio", 4, 4, 2, "mixed"), ("hubbard", 6, 2, 2, "none"),
    ("hubbard", 12, 5, 3, "mixed"), ("hubbard", 6, 4, 2, "triples")])
def test_products_match_oracle(ham, n, nu, nd, kind):
    if ham == "abinitio":
        wl = inputs.abinitio("l", n, nu, nd, n_chol=3, seed=5, n_walkers=12)
    else:
        wl = inputs.hubbard("l", n // 2, 2, nu, nd, "none", seed=5, n_walkers=12)
    wl.corr_sites = correlators(kind, n)
    rng = np.random.default_rng(8)
    wl.C = 1.0 + 0.1 * rng.standard_normal(sum(4 ** len(s) for s in wl.corr_sites))
    P = oracle.Problem(wl)
    occ = wl.init_occ.copy()
    smp, _, _ = P.sample(occ, np.zeros(wl.n_walkers, np.uint64), 91, 4, 2)
    h = V.vmc_create(wl, n_walkers=12, samples_per_walker=2, walker_precision=V.VMC_FP64, keep_fp64_store=True,
                     keep_lowp_store=True)
    V.vmc_set_params(h, wl.C, wl.f)
    V.vmc_measure(h, smp)
    x = rng.standard_normal(wl.n_params + 1)
    ref = P.lm_apply(smp, oracle.lm_factors(wl), x)
    for store, tol in ((V.VMC_STORE_FP64, 1e-10), (V.VMC_STORE_FP32, 2e-4)):
        got = V.lm_apply(h, torch.from_numpy(x).cuda(), store)
        for g, r in zip(got, ref):
            assert np.linalg.norm(g.cpu().numpy() - r) <= tol * np.linalg.norm(r)
    h.close()
