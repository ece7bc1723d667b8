// Walker kernels: Metropolis sampling from |Psi_n|^2 (Sec. II.A, fixed N and
// S_z as in Sec. III), local energy, and the per-sample derivative ratios
// O_k(n) = Psi^k_n / Psi_n of Eq. 3 for the CPS x pfaffian ansatz of Eq. 11.
//
// One warp owns one walker.  The walker keeps X = A^{-1}, A = F[occ, occ],
// in shared memory with the electron positions left unsorted (a move puts
// the new orbital in the vacated position).  For a move p -> q at position a
// with b_j = F[q, o_j] (b_a = 0):
//   Pf(A')/Pf(A) = sum_j b_j X_{ja} = -sum_j b_j X_{aj}
// (Pf is linear in row/column a; dPf/dA_aj = Pf X_{ja}).  The Jordan-Wigner
// sign of the hop cancels the sign of re-sorting the positions, so this
// unsorted ratio is the signed amplitude ratio the local energy needs.  On
// acceptance A' = A + e_a u^T - u e_a^T (u = b - A_{a,:}), whose 2x2
// Woodbury capacitance is r I, so
//   X' = X + (c y^T - y c^T) / r,  c = X_{:,a},  y = X b + e_a.
// The inverse is rebuilt from scratch (Gauss-Jordan, partial pivoting) at
// the start of every call.  The chain also multiplies up the magnitudes of its
// accepted ratios in FP64 (LogProduct), whose logarithm at a stored sample is the
// running log-amplitude that a from-scratch evaluation checks
// (vmc_sample_stats).
#include "ansatz.cuh"
#include "common.cuh"
#include "kernels.h"

namespace vmc {

struct WarpMem {
    unsigned char* base;
};


// Running product of the accepted ratios' magnitudes as m 2^e, m in [1, 2): one
// multiplication per accepted move, and one logarithm per stored sample instead
// of one per move (an FP64 logarithm is a hundred dependent instructions on a
// pipe of 16 cycles each: 40 % of an accepted move on small lattices).
struct LogProduct {
    double m = 1.0;
    int e = 0;
    __device__ __forceinline__ void mul(double x) {
        m *= fabs(x);
        const int hi = __double2hiint(m), ex = (hi >> 20) & 0x7ff;
        if (ex != 0 && ex != 0x7ff) {   // zero, denormal, infinite or NaN: left to the logarithm
            e += ex - 1023;
            m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(m));
        }
    }
    __device__ __forceinline__ double log_value() const { return log(m) + (double)e * 0.69314718055994530942; }
};

// correlator amplitude ratio C(new) / C(old): FP64 walkers multiply by the stored
// 1 / C (a division there is a dozen dependent FP64 instructions)
__device__ __forceinline__ float load_den(const DevProblem& pb, int64_t k, float) { return __ldg(pb.C32 + k); }
__device__ __forceinline__ double load_den(const DevProblem& pb, int64_t k, double) { return __ldg(pb.iC64 + k); }
__device__ __forceinline__ float ratio_of(float num, float den) { return num / den; }
__device__ __forceinline__ double ratio_of(double num, double inv) { return num * inv; }

template <typename R> struct pair_of;
template <> struct pair_of<float> { using type = float2; };
template <> struct pair_of<double> { using type = double2; };

template <typename R>
__device__ R corr_ratio_warp(const DevProblem& pb, uint32_t* cidx, int p, int q, bool commit) {
    const int lane = threadIdx.x & 31;
    int ns = pb.ns;
    int sf = p >= ns ? 2 : 1;
    int sp = p >= ns ? p - ns : p, sq = q >= ns ? q - ns : q;
    int total = (pb.site_cptr[sp + 1] - pb.site_cptr[sp]) + (pb.site_cptr[sq + 1] - pb.site_cptr[sq]);
    R prod = R(1);
    for (int base = 0; base < total; base += 32) {
        int e = base + lane;
        R r = R(1);
        int c = -1, newi = -1;
        if (e < total) {
            newi = corr_entry(pb, cidx, sp, sq, sf, e, &c);
            if (c >= 0) r = ratio_of(load_C<R>(pb, pb.corr_off[c] + newi), load_den(pb, pb.corr_off[c] + cidx[c], R(0)));
        }
        prod *= warp_prod(r);
        if (commit) {
            __syncwarp();
            if (c >= 0) cidx[c] = (uint32_t)newi;
            __syncwarp();
        }
    }
    return prod;
}

// the same by one lane, for a hop of its own
template <typename R>
__device__ R corr_ratio_hop(const DevProblem& pb, const uint32_t* cidx, int p, int q) {
    const int ns = pb.ns, sf = p >= ns ? 2 : 1;
    const int sp = p >= ns ? p - ns : p, sq = q >= ns ? q - ns : q;
    const int total = (pb.site_cptr[sp + 1] - pb.site_cptr[sp]) + (pb.site_cptr[sq + 1] - pb.site_cptr[sq]);
    R prod = R(1);
#pragma unroll 4
    for (int e = 0; e < total; ++e) {
        int c;
        const int newi = corr_entry(pb, cidx, sp, sq, sf, e, &c);
        if (c >= 0) prod *= ratio_of(load_C<R>(pb, pb.corr_off[c] + newi), load_den(pb, pb.corr_off[c] + cidx[c], R(0)));
    }
    return prod;
}

// In-place Gauss-Jordan inverse with partial pivoting of the N x N matrix X
// (row stride XS) by one warp.  col: N scratch, piv: N row indices.  Returns
// false if a pivot column is entirely zero or not finite.
template <typename R>
__device__ bool gj_invert_warp(R* X, int N, int XS, R* col, uint8_t* piv) {
    const int lane = threadIdx.x & 31;
    for (int k = 0; k < N; ++k) {
        R best = R(-1);
        int bi = N;
        for (int i = k + lane; i < N; i += 32) {
            R v = fabs(X[i * XS + k]);
            if (v > best) { best = v; bi = i; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            R ob = __shfl_xor_sync(VMC_FULL_MASK, best, o);
            int oi = __shfl_xor_sync(VMC_FULL_MASK, bi, o);
            if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        if (!(best > R(0)) || !isfinite(best)) return false;
        if (lane == 0) piv[k] = (uint8_t)bi;
        if (bi != k) {
            for (int j = lane; j < N; j += 32) {
                R t = X[k * XS + j];
                X[k * XS + j] = X[bi * XS + j];
                X[bi * XS + j] = t;
            }
        }
        __syncwarp();
        R pinv = R(1) / X[k * XS + k];
        for (int i = lane; i < N; i += 32) col[i] = X[i * XS + k];
        __syncwarp();
        for (int j = lane; j < N; j += 32) X[k * XS + j] = (j == k ? R(1) : X[k * XS + j]) * pinv;
        __syncwarp();
        for (int j = lane; j < N; j += 32) {
            R rk = X[k * XS + j];
            for (int i = 0; i < N; ++i) {
                if (i == k) continue;
                R x = (j == k) ? R(0) : X[i * XS + j];
                X[i * XS + j] = x - col[i] * rk;
            }
        }
        __syncwarp();
    }
    for (int k = N - 1; k >= 0; --k) {
        int pk = piv[k];
        if (pk != k) {
            for (int i = lane; i < N; i += 32) {
                R t = X[i * XS + k];
                X[i * XS + k] = X[i * XS + pk];
                X[i * XS + pk] = t;
            }
        }
        __syncwarp();
    }
    return true;
}

// X = F[o, o]^{-1} for the current (unsorted) positions o, from scratch
template <typename R>
__device__ bool rebuild_inverse(const DevProblem& pb, R* X, int N, int XS, const uint8_t* pos_orb, R* col,
                                uint8_t* piv) {
    const int lane = threadIdx.x & 31;
    for (int i = 0; i < N; ++i) {
        int p = pos_orb[i];
        for (int j = lane; j < N; j += 32) X[i * XS + j] = load_F<R>(pb, p, pos_orb[j]);
    }
    __syncwarp();
    return gj_invert_warp<R>(X, N, XS, col, piv);
}

template <typename R> __device__ __forceinline__ void store_pf(const SampleArgs& a, int64_t idx, R w);
template <> __device__ __forceinline__ void store_pf<float>(const SampleArgs& a, int64_t idx, float w) {
    if (a.s_pf64) a.s_pf64[idx] = (double)w;
    if (a.s_pf32) a.s_pf32[idx] = w;
    if (a.s_pf16) a.s_pf16[idx] = __float2bfloat16_rn(w);
}
template <> __device__ __forceinline__ void store_pf<double>(const SampleArgs& a, int64_t idx, double w) {
    if (a.s_pf64) a.s_pf64[idx] = w;
    if (a.s_pf32) a.s_pf32[idx] = (float)w;
    if (a.s_pf16) a.s_pf16[idx] = __float2bfloat16_rn((float)w);
}

// One walker (or one given configuration) of the problem of `a`, run by the
// calling warp with its shared-memory slice `base`.
template <typename R>
__device__ void walker_run(const SampleArgs& a, int w, unsigned char* base) {
    const DevProblem& pb = a.pb;
    const int lane = threadIdx.x & 31;
    const int N = pb.N, M = pb.M, ns = pb.ns, nu = pb.nu, XS = a.XS;
    R* X = (R*)base;
    R* bv = X + N * XS;
    R* yv = bv + XS;
    R* cv = yv + XS;
    uint8_t* iv = (uint8_t*)yv + max(2 * XS * (int)sizeof(R), 128);   // 64 positions (yv, cv: also a queue of 32 words)
    uint32_t* cidx = (uint32_t*)(iv + 64);     // ncorr (rounded up to 4)
    uint8_t* pos_orb = (uint8_t*)(cidx + a.ncorr_pad);
    int8_t* orb_pos = (int8_t*)(pos_orb + 64); // 128

    // ---- load the configuration -----------------------------------------
    for (int o = lane; o < M; o += 32) orb_pos[o] = -1;
    __syncwarp();
    uint64_t up = 0, dn = 0;
    bool bad = false;
    for (int i = lane; i < N; i += 32) {
        int o = a.walker_occ[(int64_t)w * N + i];
        pos_orb[i] = (uint8_t)o;
        if (o >= M) bad = true;
        else if (o < ns) up |= 1ull << o;
        else dn |= 1ull << (o - ns);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        up |= __shfl_xor_sync(VMC_FULL_MASK, up, o);
        dn |= __shfl_xor_sync(VMC_FULL_MASK, dn, o);
    }
    bad = __any_sync(VMC_FULL_MASK, bad);
    if (bad || __popcll(up) != nu || __popcll(dn) != pb.nd) {
        if (lane == 0) atomicOr(a.status, ST_BAD_CONFIG);
        return;
    }
    __syncwarp();
    for (int i = lane; i < N; i += 32) orb_pos[pos_orb[i]] = (int8_t)i;
    __syncwarp();

    // ---- inverse of the pairing submatrix, from scratch -------------------
    if (!rebuild_inverse<R>(pb, X, N, XS, pos_orb, cv, iv)) {
        if (lane == 0) atomicOr(a.status, ST_SINGULAR);
        return;
    }

    // ---- correlator states --------------------------------------------------
    for (int c = lane; c < pb.ncorr; c += 32) {
        uint32_t idx = 0, wgt = 1;
        for (int j = pb.corr_ptr[c]; j < pb.corr_ptr[c + 1]; ++j) {
            int s = pb.corr_sites[j];
            idx += wgt * (uint32_t)(((up >> s) & 1ull) + 2ull * ((dn >> s) & 1ull));
            wgt <<= 2;
        }
        cidx[c] = idx;
    }
    __syncwarp();

    // row groups of the rank-2 update (FP32 keeps its order of additions, which
    // decides its chains)
    const int G = sizeof(R) == 4 || N > 32 ? 1 : N > 16 ? 2 : N > 8 ? 4 : 8;
    const uint64_t sitemask = (ns == 64) ? ~0ull : ((1ull << ns) - 1ull);
    uint64_t step = a.walker_step ? a.walker_step[w] : 0ull;
    LogProduct psi;       // |Psi| of the chain relative to its start, from the accepted ratios
    const uint32_t k0 = (uint32_t)a.seed, k1 = (uint32_t)(a.seed >> 32);
    const int n_sweeps = a.n_burn + a.spw;
    // Philox words of 32 consecutive proposals at once: lane L holds those of
    // counter step0 + L, and each proposal reads its own by shuffle (the same
    // numbers as one evaluation per proposal, a 32nd of the instructions)
    uint64_t step0 = step;
    u32x4 rl = philox4x32_10(u32x4{(uint32_t)w, (uint32_t)(step0 + lane), (uint32_t)((step0 + lane) >> 32), 0u},
                             k0, k1);

    for (int sw = 0; sw < n_sweeps; ++sw) {
        for (int t = 0; t < a.props_per_sweep; ++t) {
            if (step - step0 >= 32u) {
                step0 = step;
                const uint64_t sl = step0 + (uint64_t)lane;
                rl = philox4x32_10(u32x4{(uint32_t)w, (uint32_t)sl, (uint32_t)(sl >> 32), 0u}, k0, k1);
            }
            const int rsrc = (int)(step - step0);
            u32x4 r;
            r.x = __shfl_sync(VMC_FULL_MASK, rl.x, rsrc);
            r.y = __shfl_sync(VMC_FULL_MASK, rl.y, rsrc);
            r.z = __shfl_sync(VMC_FULL_MASK, rl.z, rsrc);
            ++step;
            int as = (int)mulhi32(r.x, (uint32_t)N);
            int p = as < nu ? nth_set_bit_warp(up, as) : ns + nth_set_bit_warp(dn, as - nu);
            int spin = p >= ns;
            uint64_t m = spin ? dn : up;
            int n_empty = ns - __popcll(m);
            if (n_empty <= 0) continue;
            int kk = (int)mulhi32(r.y, (uint32_t)n_empty);
            int q = spin * ns + nth_set_bit_warp(~m & sitemask, kk);
            R u = R(r.z >> 8) * R(1.0 / 16777216.0);
            int ap = orb_pos[p];
            // correlator factor, one membership entry per lane when the two
            // sites have at most 32: its two parameter loads (L2) go out
            // first and are waited on after the pfaffian row product
            const int csf = spin + 1, csp = p - spin * ns, csq = q - spin * ns;
            const int ctot = (pb.site_cptr[csp + 1] - pb.site_cptr[csp]) + (pb.site_cptr[csq + 1] - pb.site_cptr[csq]);
            const bool cfast = ctot <= 32;
            R cnum = R(1), cden = R(1);
            int cc = -1, cnew = -1;
            if (cfast && lane < ctot) {
                cnew = corr_entry(pb, cidx, csp, csq, csf, lane, &cc);
                if (cc >= 0) {
                    cnum = load_C<R>(pb, pb.corr_off[cc] + cnew);
                    cden = load_den(pb, pb.corr_off[cc] + cidx[cc], R(0));
                }
            }
            R acc = R(0);
            for (int j = lane; j < N; j += 32) {
                R bj = (j == ap) ? R(0) : load_F<R>(pb, q, pos_orb[j]);
                bv[j] = bj;
                acc += bj * X[ap * XS + j];
            }
            R rpf = -warp_sum(acc);
            R rc = cfast ? warp_prod(ratio_of(cnum, cden)) : corr_ratio_warp<R>(pb, cidx, p, q, false);
            R ratio = rpf * rc;
            bool accept = u < ratio * ratio;
            if (!accept) continue;
            psi.mul((double)ratio);
            __syncwarp();
            {
                // lane L owns the column pair 2L, 2L + 1 (XS even); X is
                // antisymmetric, so c = X[:, a] = -X[a, :] and
                // y_j = (X b)_j + [j = a] = -sum_i b_i X_ij + [j = a]
                using R2 = typename pair_of<R>::type;
                // FP64, N <= 32: the lanes beyond N / 2 take rows, G groups in all (an
                // FP64 instruction costs the same for 8 lanes as for 32; 64 chains of 16
                // electrons on the 4x4 lattice, 1,056 proposals each: 4,143 -> 3,043 us)
                const int cw = 32 / G, g = lane / cw, j0 = 2 * (lane % cw);
                const bool own = j0 < N;
                R2* cy = reinterpret_cast<R2*>(yv);   // (c_i / r, y_i / r) of every row
                R2 cj{R(0), R(0)}, yj{R(0), R(0)};
                const R rinv = R(1) / rpf;
                if (own) {
                    const R2 xa = *reinterpret_cast<const R2*>(X + ap * XS + j0);
                    cj.x = -xa.x;
                    cj.y = -xa.y;
                    for (int i = g; i < N; i += G) {
                        const R bi = bv[i];
                        const R2 x = *reinterpret_cast<const R2*>(X + i * XS + j0);
                        yj.x = fma(-bi, x.x, yj.x);
                        yj.y = fma(-bi, x.y, yj.y);
                    }
                }
                for (int o = cw; o < 32; o <<= 1) {
                    yj.x += __shfl_xor_sync(VMC_FULL_MASK, yj.x, o);
                    yj.y += __shfl_xor_sync(VMC_FULL_MASK, yj.y, o);
                }
                if (own) {
                    if (j0 == ap) yj.x += R(1);
                    if (j0 + 1 == ap) yj.y += R(1);
                    if (g == 0) {
                        cy[j0] = R2{cj.x * rinv, yj.x * rinv};
                        if (j0 + 1 < N) cy[j0 + 1] = R2{cj.y * rinv, yj.y * rinv};
                    }
                }
                __syncwarp();
                if (own) {
                    // X_ij += (c_i y_j - y_i c_j) / r
                    // (four rows' loads ahead of their stores)
                    for (int i = g; i < N; i += 4 * G) {
                        R2 x[4], ci[4];
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const int iv4 = min(i + G * v, N - 1);
                            ci[v] = cy[iv4];
                            x[v] = *reinterpret_cast<const R2*>(X + iv4 * XS + j0);
                        }
#pragma unroll
                        for (int v = 0; v < 4; ++v)
                            if (i + G * v < N) {
                                x[v].x = fma(ci[v].x, yj.x, fma(-ci[v].y, cj.x, x[v].x));
                                x[v].y = fma(ci[v].x, yj.y, fma(-ci[v].y, cj.y, x[v].y));
                                *reinterpret_cast<R2*>(X + (i + G * v) * XS + j0) = x[v];
                            }
                    }
                }
            }
            if (cfast) {
                __syncwarp();
                if (cc >= 0) cidx[cc] = (uint32_t)cnew;
                __syncwarp();
            } else {
                corr_ratio_warp<R>(pb, cidx, p, q, true);
            }
            if (lane == 0) {
                pos_orb[ap] = (uint8_t)q;
                orb_pos[p] = -1;
                orb_pos[q] = (int8_t)ap;
            }
            if (spin) dn = (dn & ~(1ull << (p - ns))) | (1ull << (q - ns));
            else up = (up & ~(1ull << p)) | (1ull << q);
            __syncwarp();
        }
        // periodic from-scratch rebuild bounds the drift of the rank-2 updates
        if (a.refresh_every > 0 && a.props_per_sweep > 0 && (sw + 1) % a.refresh_every == 0) {
            if (!rebuild_inverse<R>(pb, X, N, XS, pos_orb, cv, iv)) {
                if (lane == 0) atomicOr(a.status, ST_SINGULAR);
                return;
            }
        }
        if (sw < a.n_burn) continue;

        // ---- measurement ----------------------------------------------------
        const int64_t s = (int64_t)w * a.spw + (sw - a.n_burn);
        double e_lane = 0.0;
        if (a.want_energy && pb.ham == 0) {   // the ab initio energy has a pass of its own (abinitio.cu)
            // a lane per open hop: (electron, entry of its site's neighbour list)
            // queue up until 32 are there, so that every lane of the pfaffian row
            // products and correlator factors works
            auto hop = [&](uint32_t en) {
                const int i = (int)(en & 255u), k = (int)(en >> 8), p = pos_orb[i];
                const int q = (p >= ns) * ns + pb.nbr_site[k];
                R d = R(0);
#pragma unroll 8
                for (int j = 0; j < N; ++j)
                    if (j != i) d += load_F<R>(pb, q, pos_orb[j]) * X[i * XS + j];
                R rc = corr_ratio_hop<R>(pb, cidx, p, q);
                // -t * (Pf ratio = -d) * rc
                e_lane += pb.nbr_t[k] * (double)(d * rc);
            };
            uint32_t* queue = reinterpret_cast<uint32_t*>(yv);   // 32 entries
            int nq = 0;
            for (int i = 0; i < N; ++i) {
                const int p = pos_orb[i], spin = p >= ns, sp = p - spin * ns;
                const uint64_t m = spin ? dn : up;
                const int k1 = pb.nbr_ptr[sp + 1];
                for (int k0 = pb.nbr_ptr[sp]; k0 < k1; k0 += 32) {
                    const int k = k0 + lane;
                    const bool open = k < k1 && !((m >> pb.nbr_site[k < k1 ? k : k0]) & 1ull);
                    const uint32_t b = __ballot_sync(VMC_FULL_MASK, open), en = (uint32_t)i | (uint32_t)k << 8;
                    const int at = nq + __popc(b & ((1u << lane) - 1u));
                    if (open && at < 32) queue[at] = en;
                    nq += __popc(b);
                    if (nq >= 32) {
                        __syncwarp();
                        const uint32_t mine = queue[lane];
                        __syncwarp();
                        if (open && at >= 32) queue[at - 32] = en;
                        nq -= 32;
                        hop(mine);
                    }
                }
            }
            __syncwarp();
            if (lane < nq) hop(queue[lane]);
            __syncwarp();
            e_lane = warp_sum(e_lane);
            e_lane += pb.U * (double)__popcll(up & dn);
            if (!isfinite(e_lane) && lane == 0) atomicOr(a.status, ST_NONFINITE);
        }
        // ascending occupation and the position of each sorted electron
        for (int i = lane; i < N; i += 32) {
            int o = i < nu ? nth_set_bit64(up, i) : ns + nth_set_bit64(dn, i - nu);
            iv[i] = (uint8_t)orb_pos[o];
            if (a.s_occ) a.s_occ[s * a.Nst + i] = (uint8_t)o;
        }
        __syncwarp();
        if (a.s_X) {   // the whole inverse and its positions' orbitals, for the ab initio energy's pass
            R* dst = (R*)a.s_X + (s - (int64_t)a.w0 * a.spw) * N * N;
            for (int t = lane; t < N * N; t += 32) dst[t] = X[(t / N) * XS + t % N];
            for (int i = lane; i < N; i += 32) a.s_pos[s * a.Nst + i] = pos_orb[i];
        }
        if (a.s_E && pb.ham == 0 && lane == 0) a.s_E[s] = e_lane;
        if (a.s_lnrun && lane == 0) a.s_lnrun[s] = psi.log_value();
        if (a.s_cidx)
            for (int c = lane; c < pb.ncorr; c += 32) a.s_cidx[s * a.ncst + c] = (cstate_t)cidx[c];
        for (int e = lane; e < pb.P; e += 32) {
            uint16_t t = pb.pairtab[e];
            int aa = t & 255, bb = t >> 8;
            store_pf<R>(a, s * a.Pst + e, X[iv[bb] * XS + iv[aa]]);
        }
        __syncwarp();
    }

    // ---- write the chain state back (ascending) ------------------------------
    if (a.write_back) {
        for (int i = lane; i < N; i += 32) {
            int o = i < nu ? nth_set_bit64(up, i) : ns + nth_set_bit64(dn, i - nu);
            a.walker_occ[(int64_t)w * N + i] = (uint8_t)o;
        }
        if (lane == 0 && a.walker_step) a.walker_step[w] = step;
    }
}

template <typename R>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 5 : 4) k_walkers(SampleArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int wid = threadIdx.x >> 5;
    const int w = blockIdx.x * (blockDim.x >> 5) + wid;
    if (w >= a.n_walkers) return;
    walker_run<R>(a, a.w0 + w, smem_raw + (size_t)wid * a.warp_bytes);
}

// Several problems (lattices of uneven size) in one launch: warp g runs
// walker g - wstart[b] of problem b, wstart[b] <= g < wstart[b + 1]; every
// warp has warp_bytes of shared memory (the largest of the problems').
template <typename R>
__global__ void __launch_bounds__(128, sizeof(R) == 4 ? 5 : 4) k_walkers_batch(const SampleArgs* __restrict__ args,
                                                          const int* __restrict__ wstart, int n,
                                                          size_t warp_bytes) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int wid = threadIdx.x >> 5;
    const int g = blockIdx.x * (blockDim.x >> 5) + wid;
    if (g >= wstart[n]) return;
    int b = 0;
    while (b + 1 < n && g >= wstart[b + 1]) ++b;
    walker_run<R>(args[b], g - wstart[b], smem_raw + (size_t)wid * warp_bytes);
}

template __global__ void k_walkers<float>(SampleArgs);
template __global__ void k_walkers<double>(SampleArgs);

// launch of the batched walker kernel from the unit that defines it
cudaError_t launch_walkers_batch(bool fp64, int blocks, int threads, size_t smem, cudaStream_t st,
                                 const SampleArgs* args, const int* wstart, int n, size_t warp_bytes) {
    auto kern = fp64 ? k_walkers_batch<double> : k_walkers_batch<float>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<blocks, threads, smem, st>>>(args, wstart, n, warp_bytes);
    return cudaGetLastError();
}

}  // namespace vmc
