"""The correlator sums on both sides of the line between a histogram per thread and
shared atomics, for correlators of one to three sites with blocks of their own and
shared ones (which keep the sums out of the pass).

Reference and tolerance as in test_gpu_pass.py.
"""
import numpy as np
import pytest

from paper_1108_0900_gb300 import inputs
from paper_1108_0900_gb300 import vmcsr as V
from test_gpu_pass import LD, U, rows, scatter

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 143, 144, 1151, 1152, 2303, 2304, 4608, 36863, 36864])
def test_products_at_the_line(n):
    wl = inputs.hubbard("c", 4, 2, 4, 4, "pair", seed=5, n_walkers=1)
    sites = [[0, 1], [2, 3], [4, 5], [1, 2, 6], [3, 4, 7], [0], [5]]
    wl.corr_sites = [np.asarray(s, np.int32) for s in sites]
    wl.corr_class = np.array([0, 0, 1, 2, 3, 4, 5], np.int32)
    wl.C = 1.0 + 0.1 * np.random.default_rng(2).standard_normal(wl.n_corr_params)
    base = inputs.draw_configs(np.random.default_rng(n), min(n, 4000), 8, 4, 4)
    cfgs = np.ascontiguousarray(base[np.arange(n) % len(base)])
    h = V.vmc_create(wl, n_walkers=n, samples_per_walker=1, walker_precision=V.VMC_FP64)
    V.vmc_set_params(h, wl.C, wl.f)
    V.vmc_measure(h, cfgs)
    nv, shift = wl.n_params, 1e-3
    vecs = np.random.default_rng(1).standard_normal((4, nv))
    idx, w, _ = rows(h, wl, V.VMC_STORE_FP64)
    mean = scatter(idx, w, np.ones(n), nv) / n
    size = scatter(idx, np.abs(w), np.ones(n), nv) / n
    for k in (1, 2, 4):
        out = V.sr_apply_S(h, torch.from_numpy(vecs[:k]).cuda(), shift).cpu().numpy()
        for j in range(k):
            t = (vecs[j][idx].astype(LD) * w).sum(1)
            ref = scatter(idx, w, t, nv) / n - mean * (mean @ vecs[j]) + shift * vecs[j]
            ta = (np.abs(vecs[j])[idx] * np.abs(w)).sum(1)
            bound = scatter(idx, np.abs(w), ta, nv) / n + size * (size @ np.abs(vecs[j])) + shift * np.abs(vecs[j])
            assert np.all(np.abs(out[j] - ref) <= 64 * U * bound)
    h.close()
