"""Measured cases of the matrix-free SR framework, through its public entry points.

A case is one call that a user's optimisation makes (or, for ``step``, the whole
iteration): sampling, measuring given configurations, the S product of each
store, the linear-method product, ln|Psi| with its adjoint.  The lattices, fillings, correlators
and sample counts are those of the repository's workloads, tests and benchmark, and ragged ones in between.

Results of the 32-bit paths (FP32 walkers, the BF16 product, the mixed solve) are
handed on in 32 bits, the precision that they are computed in; those with FP64
sums or FP64 arithmetic throughout stay in 64.
"""
import math

import numpy as np
import torch

DEV = "cuda"
U_HUBBARD = 4.0
SHIFT = 1e-3


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one FP64 product of the validation workload (4x4, pair
        # correlators, 4,096 samples); launches and the wait for the result count
        _case("product_fp64_4x4_pair", "product", lx=4, ly=4, up=8, dn=8, corr="pair", samples=4096, store="fp64", vectors=1),
        # the FP64 sampling of the same workload: few chains, many samples from each
        _case("sample_fp64_4x4_pair", "sample", lx=4, ly=4, up=8, dn=8, corr="pair", samples=4096, per_walker=64, store="fp64"),
        # the product of every inner CG iteration of the mixed solve, benchmark size
        _case("product_bf16_8x8_2x3", "product", lx=8, ly=8, up=28, dn=28, corr="2x3", samples=65536, store="bf16", vectors=1),
        # four right-hand sides at once (block CG) on a ragged problem
        _case("product4_bf16_6x6_2x2", "product", lx=6, ly=6, up=17, dn=15, corr="2x2", samples=20001, store="bf16", vectors=4),
        # the outer operator of the mixed solve on the largest sample set
        _case("product_fp32_8x8_2x2", "product", lx=8, ly=8, up=28, dn=28, corr="2x2", samples=131072, store="fp32", vectors=1),
        # the product of the plain FP64 solve, benchmark size
        _case("product_fp64_8x8_2x3", "product", lx=8, ly=8, up=28, dn=28, corr="2x3", samples=65536, store="fp64", vectors=1),
        # the headline: sampling, gradient and mixed solve of one SR iteration
        _case("step_8x8_2x3", "step", lx=8, ly=8, up=28, dn=28, corr="2x3", samples=65536, per_walker=4, store="fp32"),
        # sampling and local energy of the 24-orbital active space (singles and doubles)
        _case("sample_abinitio24", "sample", ham="abinitio", orbitals=24, up=12, dn=12, corr="all", samples=65536, per_walker=8, store="fp32"),
        # one product of the accelerated linear method on the same problem
        _case("linear_abinitio24", "linear", ham="abinitio", orbitals=24, up=12, dn=12, corr="all", samples=65536, store="fp32"),
        # the same in FP64 on a ragged set of a 4x4 lattice
        _case("linear_fp64_4x4_2x2", "linear", lx=4, ly=4, up=8, dn=8, corr="2x2", samples=4097, store="fp64"),
        # ln|Psi| of stored samples as a function of the parameters, forward and backward (autograd)
        _case("logpsi_8x8_2x2", "logpsi", lx=8, ly=8, up=28, dn=28, corr="2x2", samples=16384, store="fp64"),
        # energies and derivatives of given configurations, FP64 from scratch, with the gradient
        _case("measure_fp64_8x8_2x2", "measure", lx=8, ly=8, up=28, dn=28, corr="2x2", samples=16384, store="fp64"),
    ]


def _case(name, call, ham="hubbard", lx=0, ly=0, orbitals=0, up=0, dn=0, corr="pair", samples=0, per_walker=1,
          store="fp64", vectors=1):
    c = {"call": call, "ham": ham, "up": up, "dn": dn, "corr": corr, "samples": samples, "per_walker": per_walker,
         "store": store, "vectors": vectors}
    c.update({"orbitals": orbitals} if ham == "abinitio" else {"lx": lx, "ly": ly})
    if name:
        c["name"] = name
    return c


def draw(rng):
    call = rng.choice(["product", "product", "sample", "step", "linear", "logpsi", "measure"])

    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if call in ("sample", "linear") and rng.random() < 0.5:
        n = rng.randint(8, 24)
        up, dn = _filling(rng, n)
        kw = dict(ham="abinitio", orbitals=n, up=up, dn=dn, corr="all")
        most = 65536
    else:
        lx, ly = rng.choice([(3, 2), (4, 3), (4, 4), (5, 4), (5, 5), (6, 5), (6, 6), (7, 5), (7, 6), (8, 6), (7, 8), (8, 8)])
        up, dn = _filling(rng, lx * ly)
        corr = rng.choice(["pair", "2x2"] + (["2x3"] if lx >= 4 and ly >= 4 else []))
        kw = dict(lx=lx, ly=ly, up=up, dn=dn, corr=corr)
        most = 131072
    store = rng.choice(["bf16", "fp32", "fp64"] if call == "product" else ["fp32", "fp64"] if call in ("sample", "linear", "measure")
                       else ["fp32"] if call == "step" else ["fp64"])
    # what one pass may cost: no more than the largest listed cases
    most = {"product": 131072, "sample": min(most, 65536), "step": 65536, "linear": 65536, "logpsi": 65536, "measure": 65536}[call]
    if call in ("sample", "linear", "measure") and store == "fp64":
        most = 8192
    n_s = spread(512, most) | 1
    per = 1
    if call in ("sample", "step"):
        per = rng.choice([2, 4, 5, 8])
        n_s = max(256, n_s // per) * per
    return _case("", call, samples=n_s, per_walker=per, store=store, vectors=rng.choice([1, 1, 2, 4]) if call == "product" else 1, **kw)


def _filling(rng, n):
    """Electrons per spin: a quarter to a half of the sites, an even number in all."""
    up = rng.randint(max(1, n // 4), max(1, n // 2 - (n > 56) * 4))
    dn = max(1, up - rng.randint(0, 2))
    if (up + dn) % 2:
        dn = dn - 1 if dn > 1 else dn + 1
    return up, dn


# ---------------------------------------------------------------------------
# problems: geometry, parameters and configurations from the seed
# ---------------------------------------------------------------------------

def _problem(case, seed):
    rng = np.random.default_rng(seed)
    p = {"bonds": np.zeros((0, 2), np.int32), "h": None, "chol": None}
    if case["ham"] == "abinitio":
        n = case["orbitals"]
        p["sites"] = [np.array((i, j), np.int32) for i in range(n) for j in range(i + 1, n)]
        idx = np.arange(n)
        r = rng.standard_normal((n, n))
        p["h"] = (np.triu(r) + np.triu(r, 1).T) * np.exp(-np.abs(idx[:, None] - idx[None, :]) / 4.0)
        L = rng.standard_normal((2 * n, n, n))
        p["chol"] = 0.5 * (L + L.transpose(0, 2, 1)) * math.sqrt(2.0) / math.sqrt(2 * n)
    else:
        lx, ly = case["lx"], case["ly"]
        n = lx * ly
        at = lambda x, y: (y % ly) * lx + x % lx  # noqa: E731
        p["bonds"] = np.array([(at(x, y), b) for y in range(ly) for x in range(lx) for b in (at(x + 1, y), at(x, y + 1))], np.int32)
        if case["corr"] == "pair":
            p["sites"] = [b.copy() for b in p["bonds"]]
        else:
            px, py = int(case["corr"][0]), int(case["corr"][2])
            px, py = min(px, lx), min(py, ly)
            p["sites"] = [np.array([at(x + dx, y + dy) for dy in range(py) for dx in range(px)], np.int32) for y in range(ly) for x in range(lx)]
    p["n"] = n
    p["C"] = 1.0 + 0.01 * rng.standard_normal(sum(4 ** len(s) for s in p["sites"]))
    p["f"] = 0.1 * rng.standard_normal(2 * n * (2 * n - 1) // 2)
    p["off"] = np.cumsum([0] + [4 ** len(s) for s in p["sites"]])
    return p


def _pairing(p, dtype=torch.float64):
    """The antisymmetric pairing matrix over spin orbitals."""
    M = 2 * p["n"]
    F = torch.zeros(M, M, dtype=torch.float64, device=DEV)
    i = torch.triu_indices(M, M, 1, device=DEV)
    F[i[0], i[1]] = torch.from_numpy(p["f"]).to(DEV)
    return (F - F.T).to(dtype)


def _states(p, occ):
    """Correlator states of configurations [n, N] (ascending spin orbitals): [n, n_corr]."""
    n = p["n"]
    on = torch.zeros(occ.shape[0], 2 * n, dtype=torch.int64, device=DEV)
    on.scatter_(1, occ, 1)
    loc = on[:, :n] + 2 * on[:, n:]
    return torch.stack([sum(loc[:, int(s)] << (2 * j) for j, s in enumerate(c)) for c in p["sites"]], 1)


def _configs(case, p, count, seed):
    """Configurations near |Psi|^2: each drawn from eight uniform ones with weight |Psi|^2."""
    g = torch.Generator(DEV)
    g.manual_seed(seed)
    n, up, dn = p["n"], case["up"], case["dn"]
    F = _pairing(p, torch.float32)
    lnC = torch.from_numpy(np.log(np.abs(p["C"]))).to(DEV)
    off = torch.from_numpy(p["off"][:-1]).to(DEV)
    out = []
    for c0 in range(0, count, 16384):
        m = min(16384, count - c0)
        best, keep = None, None
        for _ in range(8):
            a = torch.rand(m, n, generator=g, device=DEV).argsort(1)[:, :up].sort(1).values
            b = torch.rand(m, n, generator=g, device=DEV).argsort(1)[:, :dn].sort(1).values + n
            occ = torch.cat([a, b], 1)
            A = F[occ[:, :, None], occ[:, None, :]]
            w = torch.linalg.slogdet(A)[1].double() + 2.0 * lnC[off + _states(p, occ)].sum(1)
            w = w - torch.log(-torch.log(torch.rand(m, generator=g, device=DEV, dtype=torch.float64)))
            if best is None:
                best, keep = w, occ
            else:
                more = w > best
                best, keep = torch.where(more, w, best), torch.where(more[:, None], occ, keep)
        out.append(keep)
    return torch.cat(out)


def _vector(size, seed):
    g = torch.Generator(DEV)
    g.manual_seed(seed + 77)
    return torch.randn(size, generator=g, device=DEV, dtype=torch.float64)


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    from paper_1108_0900_gb300 import inputs
    from paper_1108_0900_gb300 import vmcsr as V
    p = _problem(case, seed)
    wl = inputs.Workload(name="case", n_sites=p["n"], n_up=case["up"], n_dn=case["dn"],
                         ham=inputs.ABINITIO if case["ham"] == "abinitio" else inputs.HUBBARD, corr_sites=p["sites"], C=p["C"], f=p["f"],
                         bonds=p["bonds"], bond_t=np.ones(len(p["bonds"])), U=U_HUBBARD if case["ham"] == "hubbard" else 0.0,
                         h=p["h"], chol=p["chol"])
    fp64 = case["store"] == "fp64"
    per = case["per_walker"]
    h = V.vmc_create(wl, n_walkers=case["samples"] // per, samples_per_walker=per, walker_precision=V.VMC_FP64 if fp64 else V.VMC_FP32,
                     keep_fp64_store=fp64, keep_lowp_store=not fp64)
    V.vmc_set_params(h, p["C"], p["f"])
    occ = _configs(case, p, case["samples"] // per, seed).to(torch.uint8).cpu().numpy()
    store = {"fp64": V.VMC_STORE_FP64, "fp32": V.VMC_STORE_FP32, "bf16": V.VMC_STORE_BF16}[case["store"]]
    s = {"V": V, "h": h, "case": case, "store": store, "call": case["call"], "occ": occ, "seed": int(seed) + 2000, "step": 0}
    if case["call"] in ("sample", "step"):   # thermalised chains, as between two iterations
        V.vmc_set_walkers(h, occ)
        V.vmc_sample(h, 2, s["seed"])
    elif case["call"] != "measure":          # a stored set of samples
        V.vmc_measure(h, occ)
    if case["call"] == "product":
        V.sr_gradient(h, V.VMC_STORE_FP64 if fp64 else V.VMC_STORE_FP32, stats=False)
        k = case["vectors"]
        s["v"] = _vector((k, h.n_params) if k > 1 else h.n_params, seed)
    elif case["call"] == "linear":
        s["v"] = _vector(h.n_params + 1, seed)
    elif case["call"] == "logpsi":
        s["C"] = torch.from_numpy(p["C"]).to(DEV).requires_grad_()
        s["f"] = torch.from_numpy(p["f"]).to(DEV).requires_grad_()
        s["w"] = _vector(case["samples"], seed) / case["samples"]
    return s


def run(s):
    V, h, call, store = s["V"], s["h"], s["call"], s["store"]
    if call == "product":
        y = V.sr_apply_S(h, s["v"], SHIFT, store)
        return y.float() if store == V.VMC_STORE_BF16 else y
    if call == "linear":
        Hx, Sx = V.lm_apply(h, s["v"], store)
        return (Hx, Sx) if store == V.VMC_STORE_FP64 else (Hx.float(), Sx.float())
    if call == "logpsi":
        lnpsi = V.LogPsi().apply(h, s["C"], s["f"])
        return (lnpsi.detach(),) + torch.autograd.grad(lnpsi, (s["C"], s["f"]), s["w"])
    if call == "measure":
        V.vmc_measure(h, s["occ"])
    else:
        s["step"] += 1
        V.vmc_sample(h, 0, s["seed"] + s["step"])
    g, stats = V.sr_gradient(h, store)
    if store != V.VMC_STORE_FP64:
        g32, stats = g.float(), stats.astype(np.float32)
    if call == "step":
        x, _ = V.sr_cg_solve(h, g, SHIFT, 1e-6, 20000, V.VMC_CG_MIXED, allow_not_converged=True)
        return g32, stats, x.float()
    return (g, stats) if store == V.VMC_STORE_FP64 else (g32, stats)


# ---------------------------------------------------------------------------
# the work that a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    n = case["orbitals"] if case["ham"] == "abinitio" else case["lx"] * case["ly"]
    up, dn, n_s, k = case["up"], case["dn"], case["samples"], case["vectors"]
    N, M = up + dn, 2 * n
    P = N * (N - 1) // 2
    if case["corr"] == "all":
        ncorr, ncp, sites = n * (n - 1) // 2, 8 * n * (n - 1), 2
    else:
        sites = 2 if case["corr"] == "pair" else int(case["corr"][0]) * int(case["corr"][2])
        ncorr = 2 * n if case["corr"] == "pair" else n
        ncp = ncorr * 4 ** sites
    nv = ncp + M * (M - 1) // 2
    el = {"fp64": 8, "fp32": 4, "bf16": 2}[case["store"]]
    rows = n_s * (P * el + 2 * ncorr + N)          # the stored derivative ratios: values, correlator states, occupations
    product = {"bytes": rows + 16 * k * nv, "flops": 4 * k * n_s * (P + ncorr)}
    moves = up * (n - up) + dn * (n - dn)
    on_site = 2 * ncorr * sites / n                # correlators at a hop's two sites
    if case["call"] == "product":
        return product
    if case["call"] == "linear":
        # five products with the N x N inverse, the moves' correlators forward and back, the Hamiltonian's factors
        nnz = 2 * 2 * n * n * n if case["ham"] == "abinitio" else 8 * n
        return {"bytes": rows + 24 * nv, "flops": n_s * (10 * (M - N) * N * N + 8 * moves * on_site + 2 * nnz)}
    if case["call"] == "logpsi":
        return {"bytes": n_s * (N + 4 * ncorr + 16) + 24 * nv, "flops": n_s * (N ** 3 / 3 + 2 * N ** 3 + 2 * (P + ncorr))}
    if case["ham"] == "abinitio":
        pairs = up * (up - 1) // 2 * ((n - up) * (n - up - 1) // 2) + dn * (dn - 1) // 2 * ((n - dn) * (n - dn - 1) // 2) + up * dn * (n - up) * (n - dn)
        energy = 2 * M * N * N + 2 * (M - N) ** 2 * N + 30 * pairs + moves * (4 * N + on_site)
    else:
        energy = 2 * N * (2 * N + 2 * on_site)     # about two open hops per electron
    # written once: the store; the gradient reads it once
    out = {"bytes": 2 * rows + 16 * nv, "flops": n_s * (energy + 4 * (P + ncorr))}
    if case["call"] == "measure":
        out["flops"] += n_s * 2 * N ** 3
        return out
    # one sweep of N proposals per sample, about a third accepted, and one inverse per chain and call
    out["flops"] += n_s * N * (2 * N + on_site + 2 * N * N) + n_s / case["per_walker"] * 2 * N ** 3
    if case["call"] == "step":
        out["bytes"] += 100 * rows // 2            # about a hundred inner products over the 16-bit values
        out["flops"] += 100 * product["flops"]
    return out


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ---------------------------------------------------------------------------

def exact(case, seed):
    if case["call"] in ("sample", "step"):
        return None   # the chain decides which configurations are measured
    p = _problem(case, seed)
    occ = _configs(case, p, case["samples"], seed)
    n = p["n"]
    M, N, nc = 2 * n, case["up"] + case["dn"], len(p["C"])
    F, C = _pairing(p), torch.from_numpy(p["C"]).to(DEV)
    off = torch.from_numpy(p["off"][:-1]).to(DEV)
    n_s, nv = occ.shape[0], nc + M * (M - 1) // 2
    tri = torch.triu_indices(N, N, 1, device=DEV)
    per = max(64, min(16384, (1 << 28) // (N * N + 8 * len(p["sites"]) * N)))

    def rows(o):
        """Indices and values of the nonzero derivative ratios of configurations o, and the inverses."""
        A = F[o[:, :, None], o[:, None, :]]
        X = torch.linalg.inv(A)
        k = off + _states(p, o)
        a, b = o[:, tri[0]], o[:, tri[1]]
        pq = a * M - a * (a + 1) // 2 + b - a - 1
        return torch.cat([k, nc + pq], 1), torch.cat([1.0 / C[k], X[:, tri[1], tri[0]]], 1), X, A

    def chunks():
        for c in range(0, n_s, per):
            yield c, occ[c:c + per]

    if case["call"] == "product":
        v = _vector((case["vectors"], nv), seed) if case["vectors"] > 1 else _vector(nv, seed)[None]
        y, mean = torch.zeros_like(v), torch.zeros(nv, dtype=torch.float64, device=DEV)
        for _, o in chunks():
            i, w, _, _ = rows(o)
            mean.index_add_(0, i.reshape(-1), w.reshape(-1) / n_s)
        for _, o in chunks():
            i, w, _, _ = rows(o)
            for j in range(len(v)):
                t = (v[j][i] * w).sum(1) - mean @ v[j]
                y[j].index_add_(0, i.reshape(-1), (w * t[:, None]).reshape(-1) / n_s)
        y += SHIFT * v
        return (y if case["vectors"] > 1 else y[0]).cpu()
    if case["call"] == "logpsi":
        w = _vector(n_s, seed) / n_s
        grad = torch.zeros(nv, dtype=torch.float64, device=DEV)
        lnpsi = []
        for c, o in chunks():
            i, x, _, A = rows(o)
            grad.index_add_(0, i.reshape(-1), (x * w[c:c + per, None]).reshape(-1))
            lnpsi.append(0.5 * torch.linalg.slogdet(A)[1] + torch.log(C[i[:, :len(p["sites"])]].abs()).sum(1))
        return torch.cat(lnpsi).cpu(), grad[:nc].cpu(), grad[nc:].cpu()

    # moves of one electron p -> v of the same spin: amplitude ratio = correlators times G[v][a], G = F[emp, occ] A^-1
    member = torch.zeros(len(p["sites"]), n, dtype=torch.int64, device=DEV)
    for c, sites in enumerate(p["sites"]):
        for j, s in enumerate(sites):
            member[c, int(s)] = 1 << (2 * j)

    def moves(o):
        on = torch.zeros(o.shape[0], M, dtype=torch.int64, device=DEV).scatter_(1, o, 1)
        return torch.argsort(on, dim=1, descending=False, stable=True)[:, :M - N].sort(1).values

    def shifted(k, po, vi):
        """Correlator parameters after the move of an electron from po to vi (k: those before)."""
        spin = 1 + (po >= n).long()
        return k + spin[..., None] * (member.T[vi % n] - member.T[po % n])

    if case["call"] == "measure":
        g1, g2 = torch.zeros(nv, dtype=torch.float64, device=DEV), torch.zeros(nv, dtype=torch.float64, device=DEV)
        hop = torch.zeros(n, n, dtype=torch.float64, device=DEV)
        for i, j in p["bonds"]:
            hop[int(i), int(j)] -= 1.0
            hop[int(j), int(i)] -= 1.0
        hop = hop * (1 - torch.eye(n, device=DEV))
        energies = []
        for _, o in chunks():
            i, w, X, _ = rows(o)
            emp = moves(o)
            G = F[emp[:, :, None], o[:, None, :]] @ X
            t = hop[emp[:, :, None] % n, o[:, None, :] % n] * ((emp >= n)[:, :, None] == (o >= n)[:, None, :])
            s, e, a = t.nonzero(as_tuple=True)
            k = i[s, :len(p["sites"])]
            rc = (C[shifted(k, o[s, a], emp[s, e])] / C[k]).prod(1)
            E = torch.zeros(o.shape[0], dtype=torch.float64, device=DEV).index_add_(0, s, t[s, e, a] * G[s, e, a] * rc)
            E += U_HUBBARD * (torch.zeros(o.shape[0], M, dtype=torch.int64, device=DEV).scatter_(1, o, 1).reshape(-1, 2, n).prod(1).sum(1))
            g1.index_add_(0, i.reshape(-1), w.reshape(-1) / n_s)
            g2.index_add_(0, i.reshape(-1), (w * E[:, None]).reshape(-1) / n_s)
            energies.append(E)
        E = torch.cat(energies)
        var = ((E - E.mean()) ** 2).mean()
        err = torch.sqrt(var * n_s / (n_s - 1) / n_s)
        return (g2 - E.mean() * g1).cpu(), torch.stack([E.mean(), var, err]).cpu()

    # linear: (H x, S x) with H = c0 + sum_mu L_mu R_mu; each contraction with Q is linear in x, its transpose the gradient of it
    x = _vector(nv + 1, seed)
    I = torch.eye(n, dtype=torch.float64, device=DEV)
    if case["ham"] == "abinitio":
        L = torch.from_numpy(p["chol"]).to(DEV)
        kin = torch.from_numpy(p["h"]).to(DEV) - 0.5 * torch.einsum("mpq,mqs->ps", L, L)
        Lf, Rf, c0 = L * math.sqrt(0.5), L * math.sqrt(0.5), 0.0
    else:
        kin = torch.zeros(n, n, dtype=torch.float64, device=DEV)
        for i, j in p["bonds"]:
            if i != j:
                kin[int(i), int(j)] -= 1.0
                kin[int(j), int(i)] -= 1.0
        Rf = torch.diag_embed(I)
        Lf, c0 = 0.5 * U_HUBBARD * Rf, -0.5 * U_HUBBARD * N
    Lf, Rf = torch.cat([Lf, kin[None] / (2 * N), I[None]]), torch.cat([Rf, I[None], kin[None] / (2 * N)])
    Hx, Sx = torch.zeros_like(x), torch.zeros_like(x)
    up = torch.triu_indices(M, M, 1, device=DEV)
    per = max(64, min(4096, (1 << 24) // (N * (M - N) * max(1, len(p["sites"]) // 16))))
    for _, o in chunks():
        i, w, X, _ = rows(o)
        emp = moves(o)
        G = F[emp[:, :, None], o[:, None, :]] @ X
        e, a = ((emp >= n)[0][:, None] == (o >= n)[0][None, :]).nonzero(as_tuple=True)   # the same for all samples
        po, vi = o[:, a], emp[:, e]
        k0 = i[:, :len(p["sites"])]
        k1 = shifted(k0[:, None, :], po, vi)
        rc = (C[k1] / C[k0][:, None, :]).prod(2)

        def forward(z):
            xt = z[0] + (z[1:][i] * w).sum(1)
            Z = torch.zeros(M, M, dtype=torch.float64, device=DEV).index_put((up[0], up[1]), z[1 + nc:])
            Z = Z - Z.T
            D = (Z[emp[:, :, None], o[:, None, :]] - G @ Z[o[:, :, None], o[:, None, :]]) @ X
            zc = z[1:1 + nc] / C
            dl = (zc[k1] - zc[k0][:, None, :]).sum(2)
            return rc * (G[:, e, a] * (xt[:, None] + dl) + D[:, e, a]), xt

        z = x.clone().requires_grad_()
        y, xt = forward(z)
        with torch.no_grad():
            Y = torch.zeros(o.shape[0], n * n, dtype=torch.float64, device=DEV)
            Y.scatter_add_(1, (po % n) * n + vi % n, y)
            Y.scatter_add_(1, (o % n) * (n + 1), xt[:, None].expand(-1, N).contiguous())
            Zt = (Y @ Rf.reshape(len(Rf), -1).T) @ Lf.reshape(len(Lf), -1)
            zm = Zt.gather(1, (vi % n) * n + po % n)
            zd = Zt.gather(1, (o % n) * (n + 1)).sum(1) + c0 * xt
        Hx += torch.autograd.grad((y * zm).sum() + (xt * zd).sum(), z)[0] / n_s
        with torch.no_grad():
            Sx[0] += xt.sum() / n_s
            Sx[1:].index_add_(0, i.reshape(-1), (w * xt[:, None]).reshape(-1) / n_s)
    return Hx.detach().cpu(), Sx.cpu()
