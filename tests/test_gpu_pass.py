"""The passes with FP64 sums (product and gradient) at the edges of their tiles and
splits: sample counts around a tile, the smallest and largest pairing blocks, one
spin only, one to four vectors, and every store.

Reference: Eq. 7 and the means of the stored values in numpy's long double.  A parameter's
sum has at most n_s terms whose products are good to 2^-53 (FP64 store) or 2^-46
(FP32 pairs), so the result is held to 64 or 8192 unit roundoffs of the sum of
the absolute terms.
"""
import numpy as np
import pytest

from paper_1108_0900_gb300 import inputs
from paper_1108_0900_gb300 import vmcsr as V

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -53
LD = np.longdouble


def rows(h, wl, store):
    """Index and value of every nonzero derivative ratio as stored, and E_L."""
    occ, E, cs, pf = V.vmc_get_samples(h, store)
    pairs = [(a, b) for a in range(wl.n_up) for b in range(a + 1, wl.n_up)]
    pairs += [(a, b) for a in range(wl.n_up, wl.N) for b in range(a + 1, wl.N)]
    pairs += [(a, b) for a in range(wl.n_up) for b in range(wl.n_up, wl.N)]
    p = occ[:, [a for a, _ in pairs]].astype(np.int64)
    q = occ[:, [b for _, b in pairs]].astype(np.int64)
    k = wl.corr_param_off + cs.astype(np.int64)
    idx = np.concatenate([k, wl.n_corr_params + p * wl.M - p * (p + 1) // 2 + q - p - 1], 1)
    return idx, np.concatenate([1.0 / wl.C[k], pf], 1), E


def scatter(idx, w, t, nv):
    out = np.zeros(nv, LD)   # wider than FP64: the reference's own sums stay out of the bounds
    np.add.at(out, idx.ravel(), (w.astype(LD) * t.astype(LD)[:, None]).ravel())
    return out


@pytest.mark.parametrize("lx,ly,nu,nd,corr,n", [
    (2, 1, 1, 1, "none", 5), (3, 2, 2, 0, "pair", 33), (4, 2, 3, 1, "2x2", 1), (4, 4, 8, 8, "pair", 4865),
    (5, 5, 7, 9, "pair", 1000), (6, 6, 17, 15, "2x2", 31), (7, 8, 28, 26, "2x2", 913), (8, 8, 32, 32, "pair", 65),
    (8, 8, 2, 4, "2x2", 20000)])
def test_products_and_means_of_the_stored_values(lx, ly, nu, nd, corr, n):
    wl = inputs.hubbard("p", lx, ly, nu, nd, corr, seed=3, n_walkers=1)
    cfgs = inputs.draw_configs(np.random.default_rng(n), n, wl.n_sites, nu, nd)
    h = V.vmc_create(wl, n_walkers=n, samples_per_walker=1, walker_precision=V.VMC_FP64, keep_fp64_store=True,
                     keep_lowp_store=True)
    V.vmc_set_params(h, wl.C, wl.f)
    V.vmc_measure(h, cfgs)
    nv, shift = wl.n_params, 1e-3
    vecs = np.random.default_rng(1).standard_normal((4, nv))
    for store, u in ((V.VMC_STORE_FP64, 64 * U), (V.VMC_STORE_FP32, 8192 * U), (V.VMC_STORE_BF16, 64 * U)):
        idx, w, E = rows(h, wl, store)
        mean = scatter(idx, w, np.ones(n), nv) / n
        size = scatter(idx, np.abs(w), np.ones(n), nv) / n
        E = E.astype(LD)
        g_ref = scatter(idx, w, E, nv) / n - E.mean() * mean
        g, _ = V.sr_gradient(h, store)
        bound = scatter(idx, np.abs(w), np.abs(E), nv) / n + np.abs(E).mean() * size
        assert np.all(np.abs(g.cpu().numpy() - g_ref) <= u * bound)
        if store == V.VMC_STORE_BF16:
            continue   # its product has FP32 sums
        for k in (1, 2, 4):
            out = V.sr_apply_S(h, torch.from_numpy(vecs[:k]).cuda(), shift, store).cpu().numpy()
            for j in range(k):
                t = (vecs[j][idx].astype(LD) * w).sum(1)
                ref = scatter(idx, w, t, nv) / n - mean * (mean @ vecs[j]) + shift * vecs[j]
                ta = (np.abs(vecs[j])[idx] * np.abs(w)).sum(1)
                bound = scatter(idx, np.abs(w), ta, nv) / n + size * (size @ np.abs(vecs[j])) + shift * np.abs(vecs[j])
                assert np.all(np.abs(out[j] - ref) <= u * bound)
    h.close()
