// Local energy of the ab initio Hamiltonian (H of Eq. 9, fixed N and S_z) of
// the stored samples, one CTA per sample.  E_L = <n|H|n> + sum over single and
// double same-spin-conserving moves of <n|H|n'> Psi_n'/Psi_n.  With the new
// orbitals put in place of the old ones, the amplitude ratios are the
// in-place pfaffian ratios (their Jordan-Wigner signs cancel against those of
// the matrix elements, as for the hops) and the matrix elements are the
// Slater-Condon magnitudes:
//   single p->x:  h_px + sum_{k occ != p} [(px|kk) - d(s_k, s_p) (pk|kx)]
//   double p1->x, p2->y:  (p1 x|p2 y) - d(same spin) (p1 y|p2 x).
// X = A^{-1} as the walker that wrote the sample held it (the stored pairing
// block is one triangle of it).  The pfaffian ratio of a single move is
// G[x][a], G[x][j] = sum_k F[x][o_k] X[k][j]; of a double move double_ratio.
//
// Correlators of at most two sites (pairs): the correlator factor of any
// excitation is a product of the per-sample tables of ab_tables (where they hold:
// TableRange), and what an
// excitation does not share with its neighbours is a handful of shared loads,
// its integrals and a dozen multiply-adds (ab_doubles_mixed, ab_doubles_same).
//
// What bounds it: shared-memory and L1 wavefronts and the latency of the
// integral rows out of L2.  As a pass of its own with four warps per sample an
// SM holds five samples, 20 warps; one warp per sample inside the walkers'
// kernel left 12 warps per SM beside its tables and overran the instruction
// cache (24 ms).  24 orbitals, 12 + 12 electrons, 65,536 samples, FP32, with the
// sampling (2.5 ms) and the gradient: 12.2 ms; 136 ms with each excitation's
// correlator factor evaluated by itself, 700 instructions per excitation.  CTAs
// per SM, at an earlier state of the kernel: 4 14.1, 5 13.6, 6 14.0 ms.
//
// The products G and H and the pfaffian ratios keep the order and the roundings
// that they have in the positions' order of the walker: on nearly singular blocks
// E_L's FP32 rounding grows with |X|, and two orders differ by 1e-5 of the gradient's
// norm there.  FP32: the diagonal is summed in FP64, every double excitation in an
// FP32 pair.
#include "ansatz.cuh"
#include "common.cuh"
#include "kernels.h"

namespace vmc {

// Sum of many terms of the walker's precision with FP64 accuracy: FP64 for
// FP64 walkers; for FP32 walkers an FP32 pair (two-sum: the rounding error of
// each add goes to the low word), which keeps the sum off the FP64 pipe.
template <typename R> struct term_sum;
template <> struct term_sum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    // x y, or nothing (x may be infinite or NaN then)
    __device__ __forceinline__ void add_product(bool none, double x, double y) { s = fma(none ? 0.0 : x, y, s); }
    __device__ __forceinline__ double value() const { return s; }
};
template <> struct term_sum<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float s = __fadd_rn(hi, x);
        const float bx = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bx)), __fsub_rn(x, bx)));
        hi = s;
    }
    __device__ __forceinline__ void add_product(bool none, float x, float y) {
        const float p = x * y;
        add(none ? 0.f : p);
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

template <typename R> __device__ __forceinline__ R load_h(const DevProblem& pb, int i, int j);
template <> __device__ __forceinline__ float load_h<float>(const DevProblem& pb, int i, int j) {
    return __ldg(pb.h32 + i * pb.ns + j);
}
template <> __device__ __forceinline__ double load_h<double>(const DevProblem& pb, int i, int j) {
    return __ldg(pb.h64 + i * pb.ns + j);
}
// (pq|rs) over spatial orbitals
template <typename R> __device__ __forceinline__ R load_eri(const DevProblem& pb, int p, int q, int r, int s);
template <> __device__ __forceinline__ float load_eri<float>(const DevProblem& pb, int p, int q, int r, int s) {
    const int n = pb.ns;
    return __ldg(pb.eri32 + ((p * n + q) * n + r) * n + s);
}
template <> __device__ __forceinline__ double load_eri<double>(const DevProblem& pb, int p, int q, int r, int s) {
    const int n = pb.ns;
    return __ldg(pb.eri64 + ((p * n + q) * n + r) * n + s);
}

// Correlator factor of moving two electrons (p1 -> x, p2 -> y; sf = 1 up, 2
// down for each move) given the two single-move factors r1, r2: correlators
// touched by both moves hold a site of each, so they are found through the
// site-pair lists and corrected to their joint new state.
template <typename R>
__device__ R corr_ratio_double(const DevProblem& pb, const uint32_t* cidx, int p1, int x, int p2, int y, R r1, R r2) {
    const int ns = pb.ns;
    const int sf1 = p1 >= ns ? 2 : 1, sf2 = p2 >= ns ? 2 : 1;
    const int a1[2] = {p1 % ns, x % ns}, a2[2] = {p2 % ns, y % ns};
    R corr = R(1);
    for (int u = 0; u < 2; ++u)
        for (int v = 0; v < 2; ++v) {
            const int i = a1[u], j = a2[v];
            // correlators holding a site of each move: the pair list of (i, j),
            // or every correlator on the site when both moves touch it
            const int lo = i == j ? pb.site_cptr[i] : pb.pair_ptr[i * ns + j];
            const int hi = i == j ? pb.site_cptr[i + 1] : pb.pair_ptr[i * ns + j + 1];
            for (int e = lo; e < hi; ++e) {
                const int c = i == j ? pb.site_corr[e] : pb.pair_corr[e];
                // counted once: skip if an earlier (u', v') combination also lies in c
                bool seen = false;
                for (int w = 0; w < u * 2 + v && !seen; ++w) {
                    const int i2 = a1[w >> 1], j2 = a2[w & 1];
                    seen = site_weight_in(pb, c, i2) != 0 && (i2 == j2 || site_weight_in(pb, c, j2) != 0);
                }
                if (seen) continue;
                const int old = (int)cidx[c];
                const int d1 = sf1 * (site_weight_in(pb, c, a1[1]) - site_weight_in(pb, c, a1[0]));
                const int d2 = sf2 * (site_weight_in(pb, c, a2[1]) - site_weight_in(pb, c, a2[0]));
                const int64_t o = pb.corr_off[c];
                const R c0 = load_C<R>(pb, o + old);
                corr *= load_C<R>(pb, o + old + d1 + d2) * c0 / (load_C<R>(pb, o + old + d1) * load_C<R>(pb, o + old + d2));
            }
        }
    return r1 * r2 * corr;
}

__device__ __forceinline__ int site_state(uint64_t up, uint64_t dn, int s) {
    return (int)((up >> s) & 1ull) + 2 * (int)((dn >> s) & 1ull);
}

// Factors of the sites' local states: rsite[4 s + v] = product over the correlators
// on site s of C(s in state v) / C(now), all other sites as they are.
template <typename R>
__device__ __forceinline__ void site_factors(const DevProblem& pb, R* rsite, const uint32_t* cidx, uint64_t up, uint64_t dn) {
    for (int t = threadIdx.x; t < 4 * pb.ns; t += blockDim.x) {
        const int s = t >> 2, v = t & 3, n = site_state(up, dn, s);
        R f = R(1);
        if (v != n)
            for (int ent = pb.site_cptr[s]; ent < pb.site_cptr[s + 1]; ++ent) {
                const int c = pb.site_corr[ent];
                const int64_t k = pb.corr_off[c] + (int64_t)cidx[c];
                f *= load_C<R>(pb, k + pb.site_w[ent] * (v - n)) / load_C<R>(pb, k);
            }
        rsite[t] = f;
    }
}

// Correlator factor, for correlators of at most two sites, of a move that changes
// the local state of site S[k] by D[k], k < n (repeated sites add up): the sites'
// factors, and per correlator on two of them C(both) C(now) / (C(one) C(other)).
// Only states before and after the move enter.
template <typename R, int n>
__device__ R site_move_factor(const DevProblem& pb, const uint32_t* cidx, const R* rsite, uint64_t up, uint64_t dn,
                              int (&S)[n], int (&D)[n]) {
#pragma unroll
    for (int k = 1; k < n; ++k)
#pragma unroll
        for (int m = 0; m < k; ++m)
            if (S[k] == S[m]) {
                D[m] += D[k];
                D[k] = 0;   // (a later equal site adds to the first of its kind)
                break;
            }
    R f = R(1);
#pragma unroll
    for (int k = 0; k < n; ++k)
        if (D[k] != 0) f *= rsite[4 * S[k] + site_state(up, dn, S[k]) + D[k]];
#pragma unroll
    for (int k = 0; k < n; ++k)
#pragma unroll
        for (int m = k + 1; m < n; ++m) {
            if (D[k] == 0 || D[m] == 0) continue;
            const int st = S[k] * pb.ns + S[m];
            for (int e = pb.pair_ptr[st]; e < pb.pair_ptr[st + 1]; ++e) {
                const int c = pb.pair_corr[e];
                const int64_t o = pb.corr_off[c] + (int64_t)cidx[c];
                const int dk = site_weight_in(pb, c, S[k]) * D[k], dm = site_weight_in(pb, c, S[m]) * D[m];
                f *= load_C<R>(pb, o + dk + dm) * load_C<R>(pb, o) / (load_C<R>(pb, o + dk) * load_C<R>(pb, o + dm));
            }
        }
    return f;
}

// Magnitudes that the tables of ab_tables may hold: with toggle factors within
// 2^+-kToggle and corrections within 2^+-kCorrection the product of an excitation,
// at most four of the former and six of the latter, stays a normal number at
// every step.  An excitation of moderate factor may pass through toggles that are
// not (two electrons of a site moved together where single occupancy is
// projected out), so a sample beyond goes the general way.
template <typename R> struct TableRange;
template <> struct TableRange<float> { static constexpr int kToggle = 20, kCorrection = 7; };      // 122 of 126
template <> struct TableRange<double> { static constexpr int kToggle = 200, kCorrection = 30; };   // 980 of 1022
__device__ __forceinline__ bool beyond(float v, int lim) {   // zero, infinite and NaN too
    return (uint32_t)(((__float_as_int(v) >> 23) & 255) - (127 - lim)) > 2u * (uint32_t)lim;
}
__device__ __forceinline__ bool beyond(double v, int lim) {
    return (uint32_t)(((__double2hiint(v) >> 20) & 0x7ff) - (1023 - lim)) > 2u * (uint32_t)lim;
}

template <typename R> __device__ __forceinline__ const R* eri_table(const DevProblem& pb);
template <> __device__ __forceinline__ const float* eri_table<float>(const DevProblem& pb) { return pb.eri32; }
template <> __device__ __forceinline__ const double* eri_table<double>(const DevProblem& pb) { return pb.eri64; }

// four values read as one 16-byte word (two for doubles)
template <typename R> struct alignas(16) Quad { R x, y, z, w; };
// an int carried as the bits of a word
__device__ __forceinline__ int word_int(float w) { return __float_as_int(w); }
__device__ __forceinline__ int word_int(double w) { return __double2loint(w); }
__device__ __forceinline__ float int_word(float, int i) { return __int_as_float(i); }
__device__ __forceinline__ double int_word(double, int i) { return __hiloint2double(0, i); }

// Pfaffian ratio of the double move a -> x, b -> y (orbitals p1 -> x, p2 ->
// y): the second replacement on the rank-2-updated inverse, written out in G,
// X, F and H[y][x] = sum_j F[y][o_j] G[x][j].  ab_doubles_mixed evaluates the same
// operations with those of b or y alone taken out of the pair loop: on nearly
// singular blocks terms of order |X|^2 cancel down to |X|, and the shorter
// identity G G - G G + X (F - H) rounds differently there.
template <typename R>
__device__ __forceinline__ R double_ratio(R gxa, R gxb, R gya, R gyb, R xab, R xba, R fya, R fyb, R fyx, R fxa, R h) {
    const R t1 = fma(fyx, xab, fma(-fya, xab, gyb));
    const R sc = fma(-fyb, xba, gya);
    const R yb = fma(fxa, xab, -gxb);
    const R sy = fma(fyx, R(1) - gxa, fma(fxa, fma(-fyb, xab, -gya), -fma(-fyb, gxb, fma(-fya, gxa, h))));
    return fma(-sy, xba, fma(gxa, t1, sc * yb));
}

// Second moves per lane of the mixed double excitations, hole pairs per lane of those
// of one spin: what 24 orbitals with 12 + 12 electrons need in one round of the
// registers; smaller problems leave slots empty (launch_ab), larger ones take rounds.
constexpr int kAbSlots = 5;
constexpr int kAbPairSlots = 3;

// The correlator factors of a sample's excitations for correlators of at most
// two sites (the pair correlators of the ab initio ansatz), as tables over
// toggles of one spin orbital (an electron removed or added):
//   rup[s], rdn[s][u] the factor of toggling s's up spin; of its down spin with
//                    the up spin as it is (u = 0) or toggled (u = 1);
//   gss[t][s]        pair correction C(11) C(00) / (C(10) C(01)) of toggling
//                    the same spin on s and t (1 = toggled), 0 for s = t: built
//                    for one spin at a time (ab_same_spin);
//   g0[t][s]         the same for the down spin of s and the up spin of t;
//   g1[s][t]         rdn[s][1] times the same with s's up spin toggled, s an up
//                    electron and t an up hole, then s the hole and t the electron;
//   t2[b][y][u, v]   the same for the down spins of electron b and hole y
//                    with their up spins as they are (0) or toggled (1).
// One thread takes one site pair: its correlator's 16 amplitudes A[i][j] =
// C(n_s ^ i, n_t ^ j) give all entries of the pair.
template <typename F>
__device__ __forceinline__ void for_site_pairs(int ns, F f) {
    int s = 0, t = 1 + (int)threadIdx.x;   // s < t in row-major order, a CTA's threads per step
    for (int k = threadIdx.x; k < ns * (ns - 1) / 2; k += blockDim.x) {
        while (t >= ns) {
            t = t - ns + s + 2;
            ++s;
        }
        f(s, t);
        t += blockDim.x;
    }
}

// Returns whether an entry of the thread's is beyond TableRange.
template <typename R>
__device__ bool ab_tables(const DevProblem& pb, const AbLayout& L, R* tab, const uint32_t* cidx,
                          const int8_t* orb_pos, const int8_t* eidx, uint64_t up, uint64_t dn) {
    constexpr int kT = TableRange<R>::kToggle, kC = TableRange<R>::kCorrection;
    bool out = false;
    const int ns = pb.ns, nu = pb.nu, eu = ns - nu, ed = ns - pb.nd;
    R *rup = tab + L.rup, *rdn = tab + L.rdn, *g0 = tab + L.g0, *g1 = tab + L.g1, *t2 = tab + L.t2;
    R* rsite = t2;   // the factors of site s in every local state, until t2 is built
    site_factors<R>(pb, rsite, cidx, up, dn);
    for (int s = threadIdx.x; s < ns; s += blockDim.x) g0[s * ns + s] = R(1);
    __syncthreads();
    for (int t = threadIdx.x; t < 2 * ns; t += blockDim.x) {
        const int s = t >> 1, n = site_state(up, dn, s) ^ (t & 1);
        const R f = rsite[4 * s + (n ^ 2)] / rsite[4 * s + n];
        rdn[t] = f;
        out |= beyond(f, kT);
        if (t & 1) {
            rup[s] = rsite[4 * s + n];
            out |= beyond(rsite[4 * s + n], kT);
        }
    }
    __syncthreads();
    for_site_pairs(ns, [&](int s, int t) {
        R a0 = R(1), a1 = R(1), b0 = R(1), b1 = R(1), d[4] = {R(1), R(1), R(1), R(1)};
        const int vs = site_state(up, dn, s), vt = site_state(up, dn, t);
        for (int e = pb.pair_ptr[s * ns + t]; e < pb.pair_ptr[s * ns + t + 1]; ++e) {
            const int c = pb.pair_corr[e];
            const int ws = site_weight_in(pb, c, s), wt = site_weight_in(pb, c, t);
            const int64_t off = pb.corr_off[c] + (int64_t)cidx[c] - ws * vs - wt * vt;
            R A[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) A[i][j] = load_C<R>(pb, off + ws * (vs ^ i) + wt * (vt ^ j));
            a0 *= A[2][1] * A[0][0] / (A[2][0] * A[0][1]);   // down of s, up of t
            a1 *= A[3][1] * A[1][0] / (A[3][0] * A[1][1]);
            b0 *= A[1][2] * A[0][0] / (A[0][2] * A[1][0]);   // down of t, up of s
            b1 *= A[1][3] * A[0][1] / (A[0][3] * A[1][1]);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    d[2 * i + j] *= A[i + 2][j + 2] * A[i][j] / (A[i + 2][j] * A[i][j + 2]);
        }
        g0[t * ns + s] = a0;
        g0[s * ns + t] = b0;
        out |= beyond(a0, kC) | beyond(b0, kC);
        const bool us = vs & 1, ut = vt & 1, ds = vs & 2, dt = vt & 2;
        if (us != ut) {
            const int a = orb_pos[us ? s : t], x = eidx[us ? t : s];
            out |= beyond(a1, kC) | beyond(b1, kC);
            g1[a * eu + x] = us ? a1 * rdn[2 * s + 1] : b1 * rdn[2 * t + 1];
            g1[nu * eu + x * nu + a] = us ? b1 * rdn[2 * t + 1] : a1 * rdn[2 * s + 1];
        }
        if (ds != dt) {
            const int b = orb_pos[(ds ? s : t) + ns] - nu, y = eidx[(ds ? t : s) + ns] - eu;
            R* q = t2 + 4 * (b * ed + y);
            out |= beyond(d[0], kC) | beyond(d[1], kC) | beyond(d[2], kC) | beyond(d[3], kC);
            q[0] = d[0];
            q[1] = ds ? d[1] : d[2];
            q[2] = ds ? d[2] : d[1];
            q[3] = d[3];
        }
    });
    __syncthreads();
    return out;
}

// (the caller synchronises)
template <typename R>
__device__ bool ab_same_spin(const DevProblem& pb, R* gss, const uint32_t* cidx, uint64_t up, uint64_t dn, int spin) {
    const int ns = pb.ns, m = spin + 1;
    bool out = false;
    for (int s = threadIdx.x; s < ns; s += blockDim.x) gss[s * ns + s] = R(0);
    for_site_pairs(ns, [&](int s, int t) {
        R g = R(1);
        const int vs = site_state(up, dn, s), vt = site_state(up, dn, t);
        for (int e = pb.pair_ptr[s * ns + t]; e < pb.pair_ptr[s * ns + t + 1]; ++e) {
            const int c = pb.pair_corr[e];
            const int64_t k = pb.corr_off[c] + (int64_t)cidx[c];
            const int ds = site_weight_in(pb, c, s) * ((vs ^ m) - vs), dt = site_weight_in(pb, c, t) * ((vt ^ m) - vt);
            g *= load_C<R>(pb, k + ds + dt) * load_C<R>(pb, k) / (load_C<R>(pb, k + ds) * load_C<R>(pb, k + dt));
        }
        gss[s * ns + t] = gss[t * ns + s] = g;
        out |= beyond(g, TableRange<R>::kCorrection);
    });
    return out;
}

// sum over the occupied k of (pq|kk) - d(spin) (pk|kq), leaving out the
// electron itself (orbital `own` of the given spin): the two-electron part of
// the matrix element of a single move p -> q.  The integrals of one (p, q) are two
// consecutive rows.
template <typename R>
__device__ __forceinline__ R coulomb_exchange(const DevProblem& pb, int p, int q, int own, uint64_t same, uint64_t other) {
    const int nk = pb.eri_nk;
    same &= ~(1ull << own);
    const R* J = (sizeof(R) == 4 ? (const R*)pb.erijk32 : (const R*)pb.erijk64) + (size_t)(p * pb.ns + q) * 2 * nk;
    R s = R(0);
    for (int k0 = 0; k0 < nk; k0 += 4) {
        const Quad<R> c = *reinterpret_cast<const Quad<R>*>(J + k0), x = *reinterpret_cast<const Quad<R>*>(J + nk + k0);
        const uint32_t a = (uint32_t)(same >> k0), b = (uint32_t)(other >> k0);
        const R cv[4] = {c.x, c.y, c.z, c.w}, xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if ((a >> j) & 1u) s += cv[j] - xv[j];
            if ((b >> j) & 1u) s += cv[j];
        }
    }
    return s;
}

// Double excitations of one up and one down electron.  A warp walks first
// moves (a, x) of the up electrons; its lanes, one per site, form the factor of
// every down toggle on top of it and the parts of the pfaffian ratio that
// belong to electron b or hole y alone; a second move is then two 16-byte
// shared loads, its correlator pair, its integral and a dozen multiply-adds.
// Every lane keeps its second moves (b, y) in registers.  W sites per lane.
template <typename R, int W, bool FULL>
__device__ __forceinline__ void ab_doubles_mixed(const DevProblem& pb, const AbLayout& L, R* tab, const R* X, int XS,
                                                 const uint8_t* occ, const int8_t* orb_pos, const uint8_t* emp,
                                                 const int8_t* eidx, uint64_t dn, term_sum<R>& sum) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int ns = pb.ns, nu = pb.nu, nd = pb.nd, eu = ns - nu, ed = ns - nd, GS = L.GS;
    if (nu * eu == 0 || nd * ed == 0) return;
    const R *G = tab + L.G, *t2 = tab + L.t2, *g1 = tab + L.g1, *s1 = tab + L.s1, *g = tab + L.g0;
    Quad<R>* ev = reinterpret_cast<Quad<R>*>(tab + L.ev + wid * L.evs);   // down electrons, then down holes
    // the lane's sites: where what changes with x lies (electron b: G[x][b], hole
    // y: H[x][y], at px + x sx), the toggle factor, the place of the vector
    const R* px[W];
    int sx[W], dst[W];
    R rb[W];
    bool el[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
        const int s = min(lane + 32 * w, ns - 1);
        el[w] = (dn >> s) & 1ull;
        const int i = el[w] ? orb_pos[s + ns] : eidx[s + ns];
        px[w] = el[w] ? G + i : tab + L.H[1] + i - eu;
        sx[w] = el[w] ? GS : ed;
        dst[w] = el[w] ? i - nu : nd + i - eu;
        rb[w] = tab[L.rdn + 2 * s];
    }
    const int xm = (eu + 1) / 2;   // a warp's unit of work: one a, half of the x
    for (int c0 = 0; c0 < nd * ed; c0 += 32 * kAbSlots) {
        // the lane's second moves (b, y): the integral column, G[y][b], F[y][o_b];
        // slots past the end read an integral of zero
        int sb[kAbSlots], sy[kAbSlots], col[kAbSlots];
        R gyb[kAbSlots], fyb[kAbSlots];
#pragma unroll
        for (int u = 0; u < kAbSlots; ++u) {
            const int t = min(c0 + 32 * u + lane, nd * ed - 1);
            sb[u] = t / ed;
            sy[u] = t - sb[u] * ed;
            const int ob = occ[nu + sb[u]], oy = emp[eu + sy[u]];
            col[u] = (ob - ns) * ns + oy - ns;
            gyb[u] = G[(eu + sy[u]) * GS + nu + sb[u]];
            fyb[u] = load_F<R>(pb, oy, ob);
        }
        for (int un = wid; un < 2 * nu; un += nw) {
            const int a = un >> 1, xe = un & 1 ? eu : xm, i1 = occ[a];
            // what the ratio takes from (a; b, y); F[y][a] = -F[a][y], row by row
            R xab[kAbSlots], xba[kAbSlots], c1[kAbSlots], c2[kAbSlots], c3[kAbSlots];
#pragma unroll
            for (int u = 0; u < kAbSlots; ++u) {
                const R gya = G[(eu + sy[u]) * GS + a];
                xab[u] = X[a * XS + nu + sb[u]];
                xba[u] = X[(nu + sb[u]) * XS + a];
                c1[u] = fma(load_F<R>(pb, i1, emp[eu + sy[u]]), xab[u], gyb[u]);
                c2[u] = fma(-fyb[u], xba[u], gya);
                c3[u] = fma(-fyb[u], xab[u], -gya);
            }
            R ua[W], ra[W];
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const int s = min(lane + 32 * w, ns - 1);
                ua[w] = el[w] ? X[a * XS + nu + dst[w]] : -load_F<R>(pb, i1, s + ns);
                ra[w] = rb[w] * g[i1 * ns + s];
            }
            for (int x = un & 1 ? xm : 0; x < xe; ++x) {
                R hm[kAbSlots];
                const int jx = emp[x];
                const R* row = eri_table<R>(pb) + (i1 * ns + jx) * ns * ns;
#pragma unroll
                for (int u = 0; u < kAbSlots; ++u) hm[u] = c0 + 32 * u + lane < nd * ed ? __ldg(row + col[u]) : R(0);
                const R gxa = G[x * GS + a], fxa = load_F<R>(pb, jx, i1), omr = R(1) - gxa, rs = s1[a * eu + x];
                __syncwarp();   // the last first move's vectors are read
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const int s = lane + 32 * w;
                    if (s < ns) {
                        const R v = px[w][x * sx[w]], fyx = -load_F<R>(pb, jx, s + ns);
                        R r = ra[w] * g[jx * ns + s];
                        int code = 0;
                        if (s == i1 || s == jx) {
                            r = g1[s == i1 ? a * eu + x : nu * eu + x * nu + a];
                            code = el[w] ? 2 : 1;
                        }
                        // electron b: G[x][b], the factor of sc; hole y: F[y][x], its part of sy
                        Quad<R> q;
                        q.x = el[w] ? v : fyx;
                        q.y = fma(el[w] ? fxa : -gxa, ua[w], el[w] ? -v : v);
                        q.z = el[w] ? r * rs : r;   // with electron b: the first move's own factor
                        q.w = int_word(r, code);
                        ev[dst[w]] = q;
                    }
                }
                __syncwarp();
#pragma unroll
                for (int u = 0; u < kAbSlots; ++u) {
                    if (!FULL && c0 + 32 * u >= nd * ed) break;   // the warp's slot is past the end
                    const Quad<R> B = ev[sb[u]], Y = ev[nd + sy[u]];
                    const R t1 = fma(Y.x, xab[u], c1[u]);
                    const R sv = fma(Y.x, omr, fma(fxa, c3[u], -fma(-fyb[u], B.x, Y.y)));
                    const R rpf = fma(-sv, xba[u], fma(gxa, t1, c2[u] * B.y));
                    const int t = min(c0 + 32 * u + lane, nd * ed - 1);
                    // (a vanishing integral's ratio may overflow)
                    sum.add_product(hm[u] == R(0), hm[u] * rpf, B.z * Y.z * t2[4 * t + word_int(B.w) + word_int(Y.w)]);
                }
            }
        }
    }
}

// Double excitations of two electrons of one spin.  A warp walks electron pairs
// a < b, its lanes keep hole pairs x < y in registers; per electron pair the
// lanes, one per hole, form the factor of the hole's toggle on top of the two
// removed electrons.  Rows of integrals: (a x|b y) and, by the pair symmetry,
// (a y|b x) = (b x|a y), so a load touches the few rows of the lanes' x.
template <typename R, bool FULL>
__device__ __forceinline__ void ab_doubles_same(const DevProblem& pb, const AbLayout& L, R* tab, const R* X, int XS,
                                                const uint8_t* occ, const uint8_t* emp, int sp, term_sum<R>& sum) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int ns = pb.ns, GS = L.GS, n3 = ns * ns * ns;
    const int a0 = sp ? pb.nu : 0, na = sp ? pb.nd : pb.nu, x0 = sp ? ns - pb.nu : 0, nx = ns - na, o = sp ? ns : 0;
    const int npair = nx * (nx - 1) / 2;
    if (na < 2 || npair == 0) return;
    const R *G = tab + L.G, *gss = tab + L.gss, *H = tab + L.H[2 * sp];
    const R* rt = sp ? tab + L.rdn : tab + L.rup;
    const int rs = sp ? 2 : 1;
    Quad<R>* ev = reinterpret_cast<Quad<R>*>(tab + L.ev + wid * L.evs);   // holes: G[h][a], G[h][b], F[h][a], F[h][b]
    R* er = reinterpret_cast<R*>(ev + nx);                                  // and their toggle factors
    for (int c0 = 0; c0 < npair; c0 += 32 * kAbPairSlots) {
        int sx[kAbPairSlots], sy[kAbPairSlots], col[kAbPairSlots];
        R fyx[kAbPairSlots], h[kAbPairSlots], gxy[kAbPairSlots];
        {
            int x = 0, y = 1 + c0 + lane;   // hole pairs x < y in row-major order
#pragma unroll
            for (int u = 0; u < kAbPairSlots; ++u) {
                while (y >= nx && x < nx - 2) {
                    y = y - nx + x + 2;
                    ++x;
                }
                const int yc = min(y, nx - 1);   // past the end: any pair, weight zero
                const int qx = emp[x0 + x], qy = emp[x0 + yc];
                sx[u] = x;
                sy[u] = yc;
                col[u] = (qx - o) * ns * ns + qy - o;
                fyx[u] = load_F<R>(pb, qy, qx);
                h[u] = H[x * nx + yc];
                gxy[u] = y < nx ? gss[(qx - o) * ns + qy - o] : R(0);
                y += 32;
            }
        }
        int a = 0, b = 1 + wid;
        while (b >= na && a < na) {
            b = b - na + a + 2;
            ++a;
        }
        while (a < na - 1) {
            const int pa = occ[a0 + a], pq = occ[a0 + b], i1 = pa - o, i2 = pq - o;
            const R *row1 = eri_table<R>(pb) + i1 * n3 + i2 * ns, *row2 = eri_table<R>(pb) + i2 * n3 + i1 * ns;
            R hm[kAbPairSlots], hx[kAbPairSlots];
#pragma unroll
            for (int u = 0; u < kAbPairSlots; ++u) {
                hm[u] = __ldg(row1 + col[u]);
                hx[u] = __ldg(row2 + col[u]);
            }
            const R xab = X[(a0 + a) * XS + a0 + b], xba = X[(a0 + b) * XS + a0 + a];
            const R rab = rt[rs * i1] * rt[rs * i2] * gss[i1 * ns + i2];
            __syncwarp();   // the last electron pair's vectors are read
            for (int k = lane; k < nx; k += 32) {
                const int q = emp[x0 + k], s = q - o;
                ev[k] = Quad<R>{G[(x0 + k) * GS + a0 + a], G[(x0 + k) * GS + a0 + b], -load_F<R>(pb, pa, q),
                                -load_F<R>(pb, pq, q)};
                er[k] = rt[rs * s] * gss[i1 * ns + s] * gss[i2 * ns + s];
            }
            __syncwarp();
#pragma unroll
            for (int u = 0; u < kAbPairSlots; ++u) {
                if (!FULL && c0 + 32 * u >= npair) break;   // the warp's slot is past the end
                const Quad<R> Vx = ev[sx[u]], Vy = ev[sy[u]];
                const R rpf = double_ratio<R>(Vx.x, Vx.y, Vy.x, Vy.y, xab, xba, Vy.z, Vy.w, fyx[u], Vx.z, h[u]);
                const R d = hm[u] - hx[u];
                sum.add_product(d == R(0), d * rpf, er[sx[u]] * er[sy[u]] * gxy[u] * rab);
            }
            b += nw;
            while (b >= na && a < na) {
                b = b - na + a + 2;
                ++a;
            }
        }
    }
}

template <typename R, int W, bool FULL>
__global__ void __launch_bounds__(kAbThreads, sizeof(R) == 4 ? 5 : 3) k_ab_energy(AbArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double red[kAbThreads / 32];
    const DevProblem& pb = a.pb;
    const int tid = threadIdx.x, bd = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = bd >> 5;
    const int ns = pb.ns, M = pb.M, N = pb.N, nu = pb.nu, nd = pb.nd;
    const int eu = ns - nu, ed = ns - nd, E = eu + ed, XS = N | 1;
    const AbLayout L = ab_layout(ns, nu, nd, nw);
    const int GS = L.GS;
    R* tab = (R*)smem;
    R* X = tab + a.elems;                        // A^{-1}
    uint32_t* cidx = (uint32_t*)(X + N * XS);
    uint8_t* occ = (uint8_t*)(cidx + pb.ncorr);
    uint8_t* emp = occ + 64;
    int8_t* orb_pos = (int8_t*)(emp + 128);
    int8_t* eidx = orb_pos + 128;
    R *G = tab + L.G, *Rs = tab + L.g0;          // Rs: the general path's single-move or site factors
    const uint64_t smask = (ns == 64) ? ~0ull : ((1ull << ns) - 1ull);

    for (int64_t s = blockIdx.x; s < a.n_s; s += gridDim.x) {
        // configuration; a sample that was never written (its walker failed) is
        // left alone, the walker has set the status; positions and correlator
        // states are written together, so where the positions hold, so do the states
        uint64_t up = 0, dn = 0;
        bool bad = false;
        for (int i = 0; i < N; ++i) {
            const int o = a.pos[s * a.Nst + i];
            if (tid == 0) occ[i] = (uint8_t)o;
            bad = bad || o >= M;
            if (o < ns) up |= 1ull << o;
            else dn |= 1ull << ((o - ns) & 63);
        }
        if (bad || __popcll(up) != nu || __popcll(dn) != nd) continue;   // the same in every thread
        for (int c = tid; c < pb.ncorr; c += bd) cidx[c] = a.s_cidx[s * a.ncst + c];
        for (int o = tid; o < M; o += bd) {
            // an empty orbital's rank among those of its spin
            const bool d = o >= ns;
            const int so = d ? o - ns : o;
            const uint64_t m = d ? dn : up;
            if (!((m >> so) & 1ull)) {
                const int h = (d ? eu : 0) + __popcll(~m & ((1ull << so) - 1ull));
                eidx[o] = (int8_t)h;
                emp[h] = (uint8_t)o;
            }
        }
        for (int i = tid; i < N; i += bd) orb_pos[a.pos[s * a.Nst + i]] = (int8_t)i;
        const R* Xs = (const R*)a.X + s * N * N;
        for (int t = tid; t < N * N; t += bd) X[(t / N) * XS + t % N] = Xs[t];
        __syncthreads();
        // G: a warp's lanes over the electrons (W per lane), four holes per pass over X; the
        // lanes hold the holes' F rows and hand them round by shuffle
        for (int h0 = 4 * wid; h0 < E; h0 += 4 * nw) {
            R acc[4][2];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u][0] = acc[u][1] = R(0);
            for (int k0 = 0; k0 < N; k0 += 32) {
                R f[4];
                const int ok = k0 + lane < N ? occ[k0 + lane] : 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) f[u] = load_F<R>(pb, emp[min(h0 + u, E - 1)], ok);
                const int kn = min(32, N - k0);
                for (int k = 0; k < kn; ++k) {
                    const R v0 = lane < N ? X[(k0 + k) * XS + lane] : R(0);
                    const R v1 = W > 1 && lane + 32 < N ? X[(k0 + k) * XS + lane + 32] : R(0);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const R fk = __shfl_sync(VMC_FULL_MASK, f[u], k);
                        acc[u][0] = fma(fk, v0, acc[u][0]);
                        if (W > 1) acc[u][1] = fma(fk, v1, acc[u][1]);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (h0 + u < E) {
                    if (lane < N) G[(h0 + u) * GS + lane] = acc[u][0];
                    if (W > 1 && lane + 32 < N) G[(h0 + u) * GS + lane + 32] = acc[u][1];
                }
        }
        bool out = false;   // a table's entry of this thread is beyond the range
        if (a.pairs) out = ab_tables<R>(pb, L, tab, cidx, orb_pos, eidx, up, dn);
        __syncthreads();
        // H over pairs of empty orbitals y > x, by class [x][y]
        {
            int y = 1, x = tid;
            for (int t = tid; t < E * (E - 1) / 2; t += bd) {
                while (x >= y) {
                    x -= y;
                    ++y;
                }
                const int yq = emp[y];
                R acc = R(0);
                for (int j = 0; j < N; ++j) acc += load_F<R>(pb, yq, occ[j]) * G[x * GS + j];
                if (y < eu) tab[L.H[0] + x * eu + y] = acc;
                else if (x < eu) tab[L.H[1] + x * ed + y - eu] = acc;
                else tab[L.H[2] + (x - eu) * ed + y - eu] = acc;
                x += bd;
            }
        }
        double e = 0.0;
        // diagonal: sum_k h_kk + sum_{k < l} [(kk|ll) - d(s_k, s_l) (kl|lk)], the largest
        // part of E_L, in FP64
        for (int t = tid; t < N; t += bd) {
            const int k = occ[t] >= ns ? occ[t] - ns : occ[t];
            e += (double)load_h<R>(pb, k, k);
        }
        {
            const R* jk = sizeof(R) == 4 ? (const R*)pb.erijk32 : (const R*)pb.erijk64;
            int l = 1, k = tid;
            for (int t = tid; t < N * (N - 1) / 2; t += bd) {
                while (k >= l) {
                    k -= l;
                    ++l;
                }
                const int ok = occ[k], ol = occ[l], sk = ok >= ns ? ok - ns : ok, sl = ol >= ns ? ol - ns : ol;
                const R* J = jk + (size_t)(sk * ns + sk) * 2 * pb.eri_nk + sl;
                R w = J[0];
                if ((ok >= ns) == (ol >= ns)) w -= J[pb.eri_nk];
                e += (double)w;
                k += bd;
            }
        }
        term_sum<R> sum;
        double e1 = 0.0;         // singles
        bool general = !a.pairs;
        if (a.pairs) {
            R *rup = tab + L.rup, *rdn = tab + L.rdn, *gss = tab + L.gss, *s1 = tab + L.s1;
            for (int sp = 0; sp < 2; ++sp) {
                const int a0 = sp ? nu : 0, na = sp ? nd : nu, x0 = sp ? eu : 0, nx = sp ? ed : eu, o1 = sp ? ns : 0;
                __syncthreads();
                out |= ab_same_spin<R>(pb, gss, cidx, up, dn, sp);
                general = __syncthreads_or(out);
                if (general) break;
                // singles, and their correlator factors s1[a][x]
                for (int t = tid; t < na * nx; t += bd) {
                    const int ia = a0 + t / nx, ix = x0 + t % nx, p = occ[ia], q = emp[ix], sp_ = p - o1, sq = q - o1;
                    const R r = (sp ? rdn[2 * sp_] * rdn[2 * sq] : rup[sp_] * rup[sq]) * gss[sp_ * ns + sq];
                    s1[t] = r;
                    const R hm = load_h<R>(pb, sp_, sq) + coulomb_exchange<R>(pb, sp_, sq, sp_, sp ? dn : up, sp ? up : dn);
                    e1 += (double)(hm * G[ix * GS + ia] * r);
                }
                __syncthreads();
                ab_doubles_same<R, FULL>(pb, L, tab, X, XS, occ, emp, sp, sum);
                if (sp == 0) {
                    __syncwarp();
                    ab_doubles_mixed<R, W, FULL>(pb, L, tab, X, XS, occ, orb_pos, emp, eidx, dn, sum);
                }
            }
        }
        if (general) {
            // correlators of more sites, tables that do not fit or do not hold: every
            // excitation's factor by itself, from the sites' factors or (more sites)
            // those of the single moves, Rs[a][ie] (same spin only)
            const bool sites2 = pb.max_csites <= 2;
            sum = term_sum<R>();
            e1 = 0.0;
            if (sites2) site_factors<R>(pb, Rs, cidx, up, dn);
            else
                for (int t = tid; t < N * E; t += bd) {
                    const int p = occ[t / E], q = emp[t % E];
                    Rs[t] = ((p >= ns) == (q >= ns)) ? corr_ratio_serial<R>(pb, cidx, p, q) : R(0);
                }
            __syncthreads();
            for (int t = tid; t < N * E; t += bd) {
                const int ia = t / E, ie = t % E;
                const int p = occ[ia], x = emp[ie];
                if ((p >= ns) != (x >= ns)) continue;
                const bool d = p >= ns;
                const int ip = d ? p - ns : p, iq = d ? x - ns : x;
                const R hm = load_h<R>(pb, ip, iq) + coulomb_exchange<R>(pb, ip, iq, ip, d ? dn : up, d ? up : dn);
                R r;
                if (sites2) {
                    int S[2] = {ip, iq}, D[2] = {d ? -2 : -1, d ? 2 : 1};
                    r = site_move_factor<R, 2>(pb, cidx, Rs, up, dn, S, D);
                } else r = Rs[t];
                e1 += (double)(hm * G[ie * GS + ia] * r);
            }
            // doubles: up-up, down-down and up-down classes.  Within a class the
            // threads run over (electron pair, empty pair) with the electron pair
            // outer; both pairs come from the host's tables (dexc), the position in
            // each advancing by the CTA's threads per step.
            const int nab[3] = {nu * (nu - 1) / 2, nd * (nd - 1) / 2, nu * nd};
            const int nxy[3] = {eu * (eu - 1) / 2, ed * (ed - 1) / 2, eu * ed};
            const uint16_t* tab_ab = pb.dexc;
            const uint16_t* tab_xy = pb.dexc + nab[0] + nab[1] + nab[2];
            for (int cls = 0; cls < 3; ++cls) {
                const int nx = nxy[cls], total = nab[cls] * nx;
                if (cls > 0) {
                    tab_ab += nab[cls - 1];
                    tab_xy += nxy[cls - 1];
                }
                if (total == 0) continue;
                int kab = tid / nx, kxy = tid - (tid / nx) * nx;
                for (int t = tid; t < total; t += bd) {
                    const uint32_t ab = tab_ab[kab], xy = tab_xy[kxy];
                    kxy += bd;
                    while (kxy >= nx) {
                        kxy -= nx;
                        ++kab;
                    }
                    const int ia = (int)(ab & 255u), ib = (int)(ab >> 8), ix = (int)(xy & 255u), iy = (int)(xy >> 8);
                    const int p1 = occ[ia], p2 = occ[ib], x = emp[ix], y = emp[iy];
                    R hm = load_eri<R>(pb, p1 % ns, x % ns, p2 % ns, y % ns);
                    if (cls < 2) hm -= load_eri<R>(pb, p1 % ns, y % ns, p2 % ns, x % ns);
                    if (hm == R(0)) continue;
                    const R h = cls == 0   ? tab[L.H[0] + ix * eu + iy]
                                : cls == 1 ? tab[L.H[2] + (ix - eu) * ed + iy - eu]
                                           : tab[L.H[1] + ix * ed + iy - eu];
                    const R rpf = double_ratio<R>(G[ix * GS + ia], G[ix * GS + ib], G[iy * GS + ia], G[iy * GS + ib],
                                                  X[ia * XS + ib], X[ib * XS + ia], load_F<R>(pb, y, p1),
                                                  load_F<R>(pb, y, p2), load_F<R>(pb, y, x), load_F<R>(pb, x, p1), h);
                    R r;
                    if (sites2) {
                        const int f1 = p1 >= ns ? 2 : 1, f2 = p2 >= ns ? 2 : 1;
                        int S[4] = {p1 % ns, x % ns, p2 % ns, y % ns}, D[4] = {-f1, f1, -f2, f2};
                        r = site_move_factor<R, 4>(pb, cidx, Rs, up, dn, S, D);
                    } else r = corr_ratio_double<R>(pb, cidx, p1, x, p2, y, Rs[ia * E + ix], Rs[ib * E + iy]);
                    sum.add(hm * rpf * r);
                }
            }
        }
        e = warp_sum(e + e1 + sum.value());
        if (lane == 0) red[wid] = e;
        __syncthreads();
        if (tid == 0) {
            double v = 0.0;
            for (int w = 0; w < nw; ++w) v += red[w];
            a.s_E[s] = v;
            if (!isfinite(v)) atomicOr(a.status, ST_NONFINITE);
        }
        __syncthreads();
    }
}

template <typename R>
static cudaError_t launch_ab(const AbArgs& a, int threads, size_t smem, int nsm, cudaStream_t st) {
    // a lane takes W sites (mixed doubles) and W electrons (rows of G)
    const bool one = a.pb.ns <= 32 && a.pb.N <= 32;
    // slots past the end: a branch for each where there are many, or in FP64, whose
    // pipe takes an empty slot like a full one (16 orbitals, 8 + 8 electrons, 8,192
    // samples: FP32 895 us without and 847 with branches, FP64 1,633 and 1,042); none where
    // every slot is needed (24 orbitals, 65,536 samples, FP32: 12.16 and 12.62 ms)
    const int ed = a.pb.ns - a.pb.nd;
    auto kern = one ? k_ab_energy<R, 1, false> : k_ab_energy<R, 2, false>;
    if constexpr (sizeof(R) == 4)
        if (a.pb.nd * ed > 32 * (kAbSlots - 1)) kern = one ? k_ab_energy<R, 1, true> : k_ab_energy<R, 2, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem);
    if (e != cudaSuccess) return e;
    const int64_t res = (int64_t)nsm * (per > 0 ? per : 1);
    kern<<<(unsigned)(a.n_s < res ? a.n_s : res), threads, smem, st>>>(a);
    return cudaGetLastError();
}

// launch from the unit that defines the kernels
cudaError_t launch_ab_energy(bool fp64, const AbArgs& a, int threads, size_t smem, int nsm, cudaStream_t st) {
    return fp64 ? launch_ab<double>(a, threads, smem, nsm, st) : launch_ab<float>(a, threads, smem, nsm, st);
}

}  // namespace vmc
