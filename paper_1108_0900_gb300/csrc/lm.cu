// Accelerated linear method (Sec. II.B): the products of the matrices of
// Eq. 8 with a vector x = (x_0, x_1 .. x_nv) over the basis
// {Psi, Psi^1 .. Psi^nv}, evaluated from the stored samples by Eq. 10 with
// the Hamiltonian in the factored form of Eq. 9,
//   H = c0 + sum_mu Lhat_mu Rhat_mu,  Lhat_mu = sum_ij L^mu_ij E_ij,
//   E_ij = sum_sigma a+_{i sigma} a_{j sigma}:
//   (H x)_i = (1/n) sum_n sum_pq Q_{n q p i} z_pq(n) + c0 (S x)_i,
//   z_pq = sum_mu L^mu_pq w_mu,  w_mu = sum_rs R^mu_rs y_rs,
//   y_rs = sum_j Q_{n r s j} x_j,  Q_{n r s j} = <n| a+_r a_s |Psi^j> / Psi_n,
//   (S x)_i = (1/n) sum_n O_i(n) (x_0 + O(n) . x).
//
// One CTA owns one sample.  Q_{n r s j} is nonzero for r occupied in n and
// s = r (then Q = O_j(n), O_0 = 1) or s empty with the spin of r (then n'
// = n with the electron at r moved to s and Q = rho Psi^j_n' / Psi_n').  The
// signed amplitude ratio of the move of the electron at sorted position a
// to the empty orbital v is rho = rho_c G[v][a], G = F[:, occ] A^{-1},
// A = F[occ, occ] (the in-place pfaffian ratio, whose sign includes the
// Jordan-Wigner sign of the hop), rho_c the correlator ratio.  Contracting
// with x never forms O(n'): sum_j Q_{n r s j} x_j is the derivative of
// rho Psi_n along x, divided by Psi_n,
//   y = rho_c (G[v][a] (x_0 + O(n).x + dln rho_c) + D[v][a]),
//   D = (X[:, occ] - G X[occ, occ]) A^{-1}    (dG along x; X = the pairing
//                                               part of x as an antisymmetric
//                                               matrix),
// and the transposed contraction sum_pq Q_{n q p i} z_pq is its adjoint:
// with c_e = z_e rho_c per move e and B = Cbar A^{-T} (Cbar[v][a] = c_e),
// the pairing amplitude f_uw collects B[v][k] at (v, o_k) and -(G^T B)[l][k]
// at (o_l, o_k), antisymmetrised, plus W O(n) with W = sum of z rho over all
// moves (and the diagonal terms), and the correlators collect
// c_e G (1/C at the new state - 1/C at the old one).
//
// Per sample: (M - N) x N x N products in shared memory (D and B only between
// orbitals of one spin; D move by move when the factors reach few moves), the
// moves that some factor reaches (a Hubbard factor's are the neighbours'), two
// contractions with the factors and one atomic add per touched parameter.
// The correlator factor of a move multiplies up the single toggles of its two
// orbitals, divided once per sample (fr, fx); for correlators of at most two
// sites the adjoint needs one sum per orbital and one add per correlator and
// toggle, not one per correlator and move.  The order and the roundings of the
// 32-bit sums are those of one warp walking the moves: on nearly singular
// blocks terms of order |X|^2 cancel down to |X|, so another order would show.
//
// What bounds it: shared-memory latency and barriers (128 threads per sample,
// 64 registers, eight samples per SM at 24 orbitals); FP64: the FP64 pipe.  24
// orbitals, 12 + 12 electrons, 65,536 samples, FP32: 6.7 ms; one warp per sample
// that divided out every correlator of every move and added it with an atomic
// took 47.4 ms.  4x4 lattice, 2x2 correlators, 4,097 samples, FP64: 0.32 ms,
// 0.57 before.  Threads x CTAs per SM by registers, FP32: 128 x 4 8.1, x 6 7.5,
// x 8 6.7 ms; 256 threads 11.4, 8.6, 7.3 ms.
#include <algorithm>
#include "ansatz.cuh"
#include "common.cuh"
#include "kernels.h"

namespace vmc {

namespace {

// rounded apart: the compiler does not fuse them
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// Correlator part of the ratio for moving the electron at spin orbital p to
// q, and the derivative of its logarithm along x (xc = x_k / C_k): sum over
// the correlators that change of xc[new state] - xc[old state].  The
// correlators on p's site, then those on q's, in list order; the factor and
// difference of a correlator that holds only one of the two sites come from
// the sample's table (fr, fx: entry 2 cptr[s] + spin len(s) + e for the e-th
// correlator on site s with that spin of s toggled), or, where that does not
// fit shared memory (fr null), from the amplitudes.
template <typename R>
__device__ __forceinline__ R corr_ratio_dir(const DevProblem& pb, const uint64_t* common, const uint32_t* cidx, int p,
                                            int q, const R* xc, const R* fr, const R* fx, R* dl) {
    const int ns = pb.ns, spin = p >= ns, sf = spin + 1;
    const int sp = spin ? p - ns : p, sq = spin ? q - ns : q;
    R prod = R(1), d = R(0);
    if (!fr) {
        const int total = (pb.site_cptr[sp + 1] - pb.site_cptr[sp]) + (pb.site_cptr[sq + 1] - pb.site_cptr[sq]);
        for (int e = 0; e < total; ++e) {
            int c;
            const int newi = corr_entry(pb, cidx, sp, sq, sf, e, &c);
            if (c < 0) continue;
            const int64_t k1 = pb.corr_off[c] + newi, k0 = pb.corr_off[c] + cidx[c];
            prod *= load_C<R>(pb, k1) / load_C<R>(pb, k0);
            d += xc[k1] - xc[k0];
        }
        *dl = d;
        return prod;
    }
    const int e1 = pb.site_cptr[sp], n1 = pb.site_cptr[sp + 1] - e1, e2 = pb.site_cptr[sq], n2 = pb.site_cptr[sq + 1] - e2;
    // a correlator holding both sites moves to a state of its own
    auto both = [&](int e, R& r, R& x) {
        const int c = pb.site_corr[e1 + e];
        const int64_t k0 = pb.corr_off[c] + cidx[c], k1 = k0 - sf * pb.site_w[e1 + e] + sf * site_weight_in(pb, c, sq);
        r = load_C<R>(pb, k1) / load_C<R>(pb, k0);
        x = xc[k1] - xc[k0];
    };
    const uint64_t m1 = common[sp * ns + sq], m2 = common[sq * ns + sp];
    const int first = __ffsll((long long)m1) - 1;
    R br = R(1), bx = R(0);
    if (m1) both(first, br, bx);
    const R *r1 = fr + 2 * e1 + spin * n1, *x1 = fx + 2 * e1 + spin * n1;
    for (int e = 0; e < n1; ++e) {
        R r = r1[e], x = x1[e];
        if ((m1 >> e) & 1ull) {
            if (e != first) both(e, br, bx);
            r = br;
            x = bx;
        }
        prod *= r;
        d += x;
    }
    const R *r2 = fr + 2 * e2 + spin * n2, *x2 = fx + 2 * e2 + spin * n2;
    for (int e = 0; e < n2; ++e) {
        const bool skip = (m2 >> e) & 1ull;
        prod *= skip ? R(1) : r2[e];
        d += skip ? R(0) : x2[e];
    }
    *dl = d;
    return prod;
}

// Adjoint of the correlator ratio of one move: coef (1/C at the new state) for
// every correlator it changes; the old-state parts are summed per correlator
// in shared memory (old[c]) and leave with the sample's own O(n) term.
template <typename R>
__device__ void corr_ratio_adjoint(const DevProblem& pb, const double* invC, const uint32_t* cidx, int p, int q,
                                   double coef, double* out, R* old) {
    const int ns = pb.ns;
    const int sf = p >= ns ? 2 : 1;
    const int sp = p >= ns ? p - ns : p, sq = q >= ns ? q - ns : q;
    const int total = (pb.site_cptr[sp + 1] - pb.site_cptr[sp]) + (pb.site_cptr[sq + 1] - pb.site_cptr[sq]);
    for (int e = 0; e < total; ++e) {
        int c;
        const int newi = corr_entry(pb, cidx, sp, sq, sf, e, &c);
        if (c < 0) continue;
        const int64_t k1 = pb.corr_off[c] + newi;
        atomicAdd(out + k1, coef * __ldg(invC + k1));
        atomicAdd(old + c, (R)coef);
    }
}

// move t of the same-spin list: up electrons to up holes, then down to down
__device__ __forceinline__ void decode_move(int t, int nu, int eu, int ed, int* a, int* ie) {
    const int nup = nu * eu;
    if (t < nup) {
        *a = t / eu;
        *ie = t % eu;
    } else {
        const int u = t - nup;
        *a = nu + u / ed;
        *ie = eu + u % ed;
    }
}

// C (+)= alpha A B over the CTA with 2 x 2 register tiles per thread:
// A(i, k) = A[i sai + k sak], B(k, j) = B[k sbk + j sbj], C[i sc + j]; i < m,
// j < n, k < K.  Ragged tiles clamp their loads and skip their stores.
template <typename R>
__device__ void block_gemm(int m, int n, int K, const R* A, int sai, int sak, const R* B, int sbk, int sbj, R* C,
                           int sc, R alpha, bool accumulate) {
    const int tn = (n + 1) / 2, nt = ((m + 1) / 2) * tn;
    for (int tile = threadIdx.x; tile < nt; tile += blockDim.x) {
        const int i0 = (tile / tn) * 2, j0 = (tile % tn) * 2;
        const R *Ar[2], *Bc[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) Ar[r] = A + min(i0 + r, m - 1) * sai;
#pragma unroll
        for (int c = 0; c < 2; ++c) Bc[c] = B + min(j0 + c, n - 1) * sbj;
        R acc[2][2] = {{R(0), R(0)}, {R(0), R(0)}};
        for (int k = 0; k < K; ++k) {
            const R av[2] = {Ar[0][k * sak], Ar[1][k * sak]}, bv[2] = {Bc[0][k * sbk], Bc[1][k * sbk]};
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < 2; ++c) acc[r][c] += av[r] * bv[c];
        }
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (i0 + r < m && j0 + c < n) {
                    R* q = C + (i0 + r) * sc + j0 + c;
                    *q = accumulate ? *q + alpha * acc[r][c] : alpha * acc[r][c];
                }
    }
}

}  // namespace

LmLayout lm_layout(int ns, int nu, int nd, int n_mu, int ncorr, int nentry, int elem, bool tables) {
    LmLayout L;
    const int N = nu + nd, E = 2 * ns - N, XS = N + 1, nex = nu * (ns - nu) + nd * (ns - nd);
    auto even = [](int n) { return (n + 1) / 2 * 2; };
    L.X = 0;
    L.G = L.X + N * XS;
    L.Xo = L.G + E * XS;
    L.Pm = L.Xo + N * XS;
    L.D = L.Pm + E * XS;
    L.Y = L.D + E * XS;
    L.w = L.Y + ns * ns;
    L.cold = L.w + n_mu;
    L.rcm = L.cold + ncorr;
    L.rcm = even(L.rcm);
    L.fr = L.rcm + std::max(nex, 2 * ns * 8 / elem);   // the ratios' place takes the event sums later
    L.fx = L.fr + (tables ? 2 * nentry : 0);
    const int n = even(L.fx + (tables ? 2 * nentry : 0));
    L.cidx_bytes = n * elem;
    L.occ_bytes = L.cidx_bytes + ncorr * 4;
    L.bytes = (L.occ_bytes + N + E + 4 * ns + 15) / 16 * 16;
    return L;
}

// x -> the antisymmetric matrix of its pairing part and x_k / C_k
template <typename R>
__global__ void k_lm_prep(DevProblem pb, const double* x, R* Xt, R* xc) {
    const int64_t MM = (int64_t)pb.M * pb.M;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < MM + pb.ncp;
         t += (int64_t)gridDim.x * blockDim.x) {
        if (t < MM) {
            const int p = (int)(t / pb.M), q = (int)(t % pb.M);
            double v = 0.0;
            if (p < q) v = x[1 + pb.ncp + pb.rowbase[p] + q];
            else if (p > q) v = -x[1 + pb.ncp + pb.rowbase[q] + p];
            Xt[t] = (R)v;
        } else {
            const int64_t k = t - MM;
            xc[k] = (R)(x[1 + k] / pb.C64[k]);
        }
    }
}

template <typename R>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 4 : 3) k_lm_apply(LmArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ R xt_s, W_s;
    const DevProblem& pb = a.pb;
    const int tid = threadIdx.x, bd = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = bd >> 5;
    const int N = pb.N, M = pb.M, ns = pb.ns, nu = pb.nu, nd = pb.nd, ncorr = pb.ncorr;
    const int eu = ns - nu, ed = ns - nd, E = eu + ed;
    const int XS = N + 1, GS = N + 1, n_mu = a.n_mu, nn = ns * ns;
    const LmLayout& L = a.L;
    R* tab = (R*)smem;
    R *X = tab + L.X, *G = tab + L.G;    // A^{-1}, sorted positions; G[ie][a], rows = empty orbitals
    R* Xo = tab + L.Xo;                  // X[o_l][o_k], later G^T B
    R* Pm = tab + L.Pm;                  // X[v][o_k] - (G Xo)[v][k], later Cbar
    R* D = tab + L.D;                    // P A^{-1}, later B = Cbar A^{-T}
    R* Y = tab + L.Y;                    // y summed over spins, later z
    R *w = tab + L.w, *cold = tab + L.cold;   // old-state adjoint sums per correlator
    R* rcm = tab + L.rcm;                // correlator ratio of every move
    R *fr = a.tables ? tab + L.fr : nullptr, *fx = tab + L.fx;   // see corr_ratio_dir
    double* ev = (double*)rcm;           // then: sum of the coefficients of every spin orbital's moves
    uint32_t* cidx = (uint32_t*)(smem + L.cidx_bytes);
    uint8_t* occ = smem + L.occ_bytes;
    uint8_t* emp = occ + N;
    int8_t* opos = (int8_t*)(emp + E);   // position of an occupied orbital, or
    int8_t* epos = opos + M;             // of an empty one (else -1)
    const R* Xt = (const R*)a.Xt;
    const R* xc = (const R*)a.xc;
    const R* Lval = (const R*)a.Lval;
    const R* Rval = (const R*)a.Rval;
    const R* pf = (const R*)a.pf;
    const R x0 = (R)a.x[0];
    const R c0 = (R)a.c0;
    const double sc = a.inv_n;
    const int nex = nu * eu + nd * ed;
    double* Hf = a.Hx + 1 + pb.ncp;

    for (int64_t s = blockIdx.x; s < a.n_s; s += gridDim.x) {
        // ---- configuration, A^{-1}, F and x over its orbitals ---------------
        uint64_t up = 0, dn = 0;
        for (int i = 0; i < N; ++i) {
            const int o = a.s_occ[s * a.Nst + i];
            if (tid == 0) occ[i] = (uint8_t)o;
            if (o < ns) up |= 1ull << o;
            else dn |= 1ull << (o - ns);
        }
        for (int c = tid; c < ncorr; c += bd) {
            cidx[c] = (uint32_t)a.s_cidx[s * a.ncst + c];
            cold[c] = R(0);
        }
        for (int o = tid; o < M; o += bd) {
            const bool d = o >= ns;
            const int so = d ? o - ns : o;
            const uint64_t m = d ? dn : up, below = (1ull << so) - 1ull;
            const bool on = (m >> so) & 1ull;
            const int r = on ? (d ? nu : 0) + __popcll(m & below) : (d ? eu : 0) + __popcll(~m & below);
            opos[o] = on ? (int8_t)r : (int8_t)-1;
            epos[o] = on ? (int8_t)-1 : (int8_t)r;
            if (!on) emp[r] = (uint8_t)o;
        }
        for (int e = tid; e < pb.P; e += bd) {
            const uint16_t t = pb.pairtab[e];
            const int aa = t & 255, bb = t >> 8;
            const R v = pf[s * a.Pst + e];
            X[bb * XS + aa] = v;
            X[aa * XS + bb] = -v;
        }
        for (int i = tid; i < N; i += bd) X[i * XS + i] = R(0);
        for (int t = tid; t < nn; t += bd) Y[t] = R(0);
        __syncthreads();
        for (int t = tid; t < E * N; t += bd) {
            const int ie = t / N, k = t % N;
            Pm[ie * GS + k] = load_F<R>(pb, emp[ie], occ[k]);
        }
        for (int t = tid; t < N * N; t += bd) {
            const int l = t / N, k = t % N;
            Xo[l * XS + k] = Xt[occ[l] * M + occ[k]];
        }
        if (a.tables)
            for (int t = tid; t < 2 * a.nentry; t += bd) {
                // entry layout 2 cptr[site] + spin len(site) + e (the host's map)
                const int2 en = a.entries[t];   // index into the site lists, spin and site
                const int c = pb.site_corr[en.x], spin = en.y & 1, site = en.y >> 1;
                const bool on = ((spin ? dn : up) >> site) & 1ull;
                const int64_t k0 = pb.corr_off[c] + cidx[c], k1 = k0 + (on ? -1 : 1) * (spin + 1) * pb.site_w[en.x];
                fr[t] = load_C<R>(pb, k1) / load_C<R>(pb, k0);
                fx[t] = xc[k1] - xc[k0];
            }
        if (wid == 0) {   // O(n) . x
            R tau = R(0);
            for (int c = lane; c < ncorr; c += 32) tau += xc[pb.corr_off[c] + cidx[c]];
            for (int e = lane; e < pb.P; e += 32) {
                const uint16_t t = pb.pairtab[e];
                const int aa = t & 255, bb = t >> 8;
                tau += Xt[occ[aa] * M + occ[bb]] * X[bb * XS + aa];
            }
            tau = warp_sum(tau);
            if (lane == 0) xt_s = x0 + tau;    // sum_j O_j(n) x_j with O_0 = 1
        }
        __syncthreads();
        const R xt = xt_s;
        // ---- G = F[emp, occ] A^{-1} ------------------------------------------
        block_gemm<R>(E, N, N, Pm, GS, 1, X, XS, 1, G, GS, R(1), false);
        __syncthreads();
        // ---- P = X[emp, occ] - G Xo; D = P A^{-1} (dG along x) ---------------
        for (int t = tid; t < E * N; t += bd) {
            const int ie = t / N, k = t % N;
            Pm[ie * GS + k] = Xt[emp[ie] * M + occ[k]];
        }
        __syncthreads();
        block_gemm<R>(E, N, N, G, GS, 1, Xo, XS, 1, Pm, GS, R(-1), true);
        __syncthreads();
        // D where moves go (one spin), or move by move when few are needed
        if (a.dense) {
            if (eu && nu) block_gemm<R>(eu, nu, N, Pm, GS, 1, X, XS, 1, D, GS, R(1), false);
            if (ed && nd) block_gemm<R>(ed, nd, N, Pm + eu * GS, GS, 1, X + nu, XS, 1, D + eu * GS + nu, GS, R(1), false);
            __syncthreads();
        }
        // ---- forward: y over the moves that a factor reaches, and the diagonal,
        // summed over spin ------------------------------------------------------
        for (int t = tid; t < nex; t += bd) {
            int ia, ie;
            decode_move(t, nu, eu, ed, &ia, &ie);
            const int p = occ[ia], v = emp[ie], sp = p >= ns ? p - ns : p, sv = v >= ns ? v - ns : v;
            if (!a.need[sp * ns + sv]) continue;
            R dl;
            const R rc = corr_ratio_dir<R>(pb, a.common, cidx, p, v, xc, fr, fx, &dl);
            rcm[t] = rc;
            R dv = R(0);
            if (a.dense) dv = D[ie * GS + ia];
            else
                for (int k = 0; k < N; ++k) dv += Pm[ie * GS + k] * X[k * XS + ia];
            const R y = rc * (G[ie * GS + ia] * (xt + dl) + dv);
            atomicAdd(&Y[sp * ns + sv], y);
        }
        for (int i = tid; i < N; i += bd) atomicAdd(&Y[(occ[i] % ns) * (ns + 1)], xt);
        __syncthreads();
        // ---- w_mu = sum_rs R^mu_rs y_rs, z_pq = sum_mu L^mu_pq w_mu ----------
        for (int mu = wid; mu < n_mu; mu += nw) {
            const int k0 = a.Rptr[mu], k1 = a.Rptr[mu + 1];
            R acc = R(0);
            if (k1 - k0 == nn) {   // every entry: no index list
#pragma unroll 4
                for (int k = lane; k < nn; k += 32) acc += Rval[k0 + k] * Y[k];
            } else {
                for (int k = k0 + lane; k < k1; k += 32) acc += Rval[k] * Y[a.Ridx[k]];
            }
            acc = warp_sum(acc);
            if (lane == 0) w[mu] = acc;
        }
        for (int t = tid; t < E * N; t += bd) Pm[(t / N) * GS + t % N] = R(0);
        __syncthreads();
        // one thread per entry, the factors that reach it in order (products and
        // sums rounded apart); a list of every factor carries no index
        for (int t = tid; t < nn; t += bd) {
            const int n = a.Lcnt[t];
            R acc = R(0);
            if (n == n_mu) {
#pragma unroll 4
                for (int j = 0; j < n; ++j) acc = add_rn(acc, mul_rn(Lval[j * nn + t], w[j]));
            } else {
                for (int j = 0; j < n; ++j) acc = add_rn(acc, mul_rn(Lval[j * nn + t], w[a.Lmu[j * nn + t]]));
            }
            Y[t] = acc;
        }
        __syncthreads();

        // ---- backward: z over the moves --------------------------------------
        for (int t = tid; t < nex; t += bd) {
            int ia, ie;
            decode_move(t, nu, eu, ed, &ia, &ie);
            const int p = occ[ia], v = emp[ie], sp = p >= ns ? p - ns : p, sv = v >= ns ? v - ns : v;
            if (!a.need[sp * ns + sv]) continue;
            const R z = Y[sv * ns + sp];   // z_{v p}: the move p -> v
            if (z == R(0)) continue;
            const R c = z * rcm[t];
            Pm[ie * GS + ia] = c;
            if (!a.pairs)
                corr_ratio_adjoint<R>(pb, a.invC, cidx, p, v, (double)(c * G[ie * GS + ia]) * sc, a.Hx + 1, cold);
        }
        __syncthreads();
        if (wid == 0) {
            R W = R(0);
            for (int i = lane; i < N; i += 32) W += Y[(occ[i] % ns) * (ns + 1)];
            if (lane == 0) W += c0 * xt;
            for (int t = lane; t < nex; t += 32) {
                int ia, ie;
                decode_move(t, nu, eu, ed, &ia, &ie);
                W += Pm[ie * GS + ia] * G[ie * GS + ia];
            }
            W = warp_sum(W);
            if (lane == 0) W_s = W;
        }
        // pair correlators: the coefficients c G summed over every orbital's moves
        if (a.pairs)
            for (int o = tid - 32; o < M; o += bd - 32) {
                if (o < 0) break;   // warp 0 is at W
                const bool d = o >= ns;
                double v = 0.0;
                if (opos[o] >= 0) {
                    const int ia = opos[o];
                    for (int ie = d ? eu : 0; ie < (d ? E : eu); ++ie) v += (double)(Pm[ie * GS + ia] * G[ie * GS + ia]);
                } else {
                    const int ie = epos[o];
                    for (int ia = d ? nu : 0; ia < (d ? N : nu); ++ia) v += (double)(Pm[ie * GS + ia] * G[ie * GS + ia]);
                }
                ev[o] = v;
            }
        // B = Cbar A^{-T} (a row of Cbar holds moves of its own spin); G^T B
        if (eu && nu) block_gemm<R>(eu, N, nu, Pm, GS, 1, X, 1, XS, D, GS, R(1), false);
        else for (int t = tid; t < eu * N; t += bd) D[(t / N) * GS + t % N] = R(0);
        if (ed && nd) block_gemm<R>(ed, N, nd, Pm + eu * GS + nu, GS, 1, X + nu, 1, XS, D + eu * GS, GS, R(1), false);
        else for (int t = tid; t < ed * N; t += bd) D[(eu + t / N) * GS + t % N] = R(0);
        __syncthreads();
        const R W = W_s;
        block_gemm<R>(N, N, E, G, 1, GS, D, GS, 1, Xo, XS, R(1), false);
        __syncthreads();

        // ---- scatter ----------------------------------------------------------
        if (tid == 0) {
            atomicAdd(a.Hx, (double)W * sc);
            if (a.Sx) atomicAdd(a.Sx, (double)xt * sc);
        }
        for (int c = tid; c < ncorr; c += bd) {
            const int64_t k = pb.corr_off[c] + cidx[c];
            const double ic = __ldg(a.invC + k);
            double old = (double)cold[c];
            if (a.pairs) {
                // every move that toggles one of the correlator's sites: the
                // orbital's sum without its move to the other site (which
                // toggles both), at the toggled state
                const int j0 = pb.corr_ptr[c], m = pb.corr_ptr[c + 1] - j0;
                const int site[2] = {pb.corr_sites[j0], m > 1 ? pb.corr_sites[j0 + 1] : 0};
                double all = 0.0;
#pragma unroll
                for (int spin = 0; spin < 2; ++spin) {
                    const uint64_t mk = spin ? dn : up;
                    double cb = 0.0;
                    int64_t kb = 0;
                    if (m > 1) {
                        const int o0 = site[0] + spin * ns, o1 = site[1] + spin * ns;
                        const bool on0 = (mk >> site[0]) & 1ull, on1 = (mk >> site[1]) & 1ull;
                        if (on0 != on1) {
                            const int at = epos[on0 ? o1 : o0] * GS + opos[on0 ? o0 : o1];
                            cb = (double)(Pm[at] * G[at]);
                            kb = k + (spin + 1) * ((on0 ? -1 : 1) + 4 * (on1 ? -1 : 1));
                            if (cb != 0.0) atomicAdd(a.Hx + 1 + kb, cb * sc * __ldg(a.invC + kb));
                        }
                    }
                    all += cb;
                    for (int j = 0; j < m; ++j) {
                        const double v = ev[site[j] + spin * ns] - cb;
                        const int64_t k1 = k + (((mk >> site[j]) & 1ull) ? -1 : 1) * (spin + 1) * (j ? 4 : 1);
                        all += v;
                        if (v != 0.0) atomicAdd(a.Hx + 1 + k1, v * sc * __ldg(a.invC + k1));
                    }
                }
                old = all * sc;
            }
            atomicAdd(a.Hx + 1 + k, ((double)W * sc - old) * ic);
            if (a.Sx) atomicAdd(a.Sx + 1 + k, (double)xt * ic * sc);
        }
        for (int e = tid; e < pb.P; e += bd) {
            const uint16_t t = pb.pairtab[e];
            const int aa = t & 255, bb = t >> 8;
            const int64_t idx = pb.rowbase[occ[aa]] + occ[bb];
            const R xba = X[bb * XS + aa];
            atomicAdd(Hf + idx, (double)(W * xba - Xo[aa * XS + bb] + Xo[bb * XS + aa]) * sc);
            if (a.Sx) atomicAdd(a.Sx + 1 + pb.ncp + idx, (double)(xt * xba) * sc);
        }
        for (int t = tid; t < E * N; t += bd) {
            const int ie = t / N, k = t % N;
            const R b = D[ie * GS + k];
            if (b == R(0)) continue;
            const int v = emp[ie], o = occ[k];
            if (v < o) atomicAdd(Hf + pb.rowbase[v] + o, (double)b * sc);
            else atomicAdd(Hf + pb.rowbase[o] + v, -(double)b * sc);
        }
        __syncthreads();
    }
}

// diag of S over the basis (without its 0 entry, which is 1): the mean of
// O_k(n)^2 over the samples, one warp per sample
template <typename R>
__global__ void k_lm_diag(LmArgs a, double* d) {
    const DevProblem& pb = a.pb;
    const int lane = threadIdx.x & 31;
    const R* pf = (const R*)a.pf;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t s = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); s < a.n_s; s += nwarps) {
        for (int c = lane; c < pb.ncorr; c += 32) {
            const int64_t k = pb.corr_off[c] + a.s_cidx[s * a.ncst + c];
            const double ic = 1.0 / __ldg(pb.C64 + k);
            atomicAdd(d + 1 + k, ic * ic * a.inv_n);
        }
        for (int e = lane; e < pb.P; e += 32) {
            const uint16_t t = pb.pairtab[e];
            const int p = a.s_occ[s * a.Nst + (t & 255)], q = a.s_occ[s * a.Nst + (t >> 8)];
            const double v = (double)pf[s * a.Pst + e];
            atomicAdd(d + 1 + pb.ncp + pb.rowbase[p] + q, v * v * a.inv_n);
        }
    }
}

// part[b * k + j] = partial sums of V[:, j] . u over block b's slice
__global__ void __launch_bounds__(256) k_lm_dots(const double* V, int64_t ld, int k, const double* u, int64_t n,
                                                 double* part) {
    __shared__ double red[8];
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    const int64_t i0 = (int64_t)blockIdx.x * per, i1 = min(n, i0 + per);
    for (int j = 0; j < k; ++j) {
        double acc = 0.0;
        for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) acc += V[(int64_t)j * ld + i] * u[i];
        acc = warp_sum(acc);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
            part[(int64_t)blockIdx.x * k + j] = t;
        }
        __syncthreads();
    }
}

// out[j] = sum over blocks of part[b * k + j]
__global__ void k_lm_dots_reduce(const double* part, int nb, int k, double* out) {
    for (int j = threadIdx.x; j < k; j += blockDim.x) {
        double t = 0.0;
        for (int b = 0; b < nb; ++b) t += part[(int64_t)b * k + j];
        out[j] = t;
    }
}

// out = alpha out + sum_j c[j] V[:, j]
__global__ void __launch_bounds__(256) k_lm_combine(double* out, const double* V, int64_t ld, int k, const double* c,
                                                    int64_t n, double alpha) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double acc = alpha == 0.0 ? 0.0 : alpha * out[i];
        for (int j = 0; j < k; ++j) acc += c[j] * V[(int64_t)j * ld + i];
        out[i] = acc;
    }
}

// t = -r / (d + eps D), D = diag(0, 1, .., 1)
__global__ void __launch_bounds__(256) k_lm_precond(double* t, const double* r, const double* d, double eps, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        t[i] = -r[i] / (d[i] + (i > 0 ? eps : 0.0));
}

// alpha += x_{1:} / Sx0 (Sec. II.B: the update relative to the component of
// the new state along Psi in the basis orthogonalised to Psi)
__global__ void __launch_bounds__(256) k_lm_update(UpdateArgs a, const double* x, double scale) {
    const int64_t nv = a.ncp + a.npf;
    int bad = 0;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nv; k += (int64_t)gridDim.x * blockDim.x) {
        const double d = scale * x[1 + k];
        if (k < a.ncp) {
            const double c = a.C64[k] + d;
            if (c == 0.0) bad |= ST_SINGULAR;
            if (!isfinite(c)) bad |= ST_NONFINITE;
            a.C64[k] = c;
            a.C32[k] = (float)c;
            a.invC64[k] = 1.0 / c;
            a.invC32[k] = (float)(1.0 / c);
        } else {
            const uint32_t pq = a.pq_of[k - a.ncp];
            const int p = (int)(pq & 0xFFFFu), q = (int)(pq >> 16);
            const double f = a.F64[(int64_t)p * a.M + q] + d;
            if (!isfinite(f)) bad |= ST_NONFINITE;
            a.F64[(int64_t)p * a.M + q] = f;
            a.F64[(int64_t)q * a.M + p] = -f;
            a.F32[(int64_t)p * a.M + q] = (float)f;
            a.F32[(int64_t)q * a.M + p] = -(float)f;
        }
    }
    if (bad) atomicOr(a.status, bad);
}

template __global__ void k_lm_diag<double>(LmArgs, double*);
template __global__ void k_lm_diag<float>(LmArgs, double*);
template __global__ void k_lm_prep<double>(DevProblem, const double*, double*, double*);
template __global__ void k_lm_prep<float>(DevProblem, const double*, float*, float*);
template __global__ void k_lm_apply<double>(LmArgs);
template __global__ void k_lm_apply<float>(LmArgs);

}  // namespace vmc
