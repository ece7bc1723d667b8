// FP64 evaluation of given configurations from scratch, one warp per sample:
// the pairing inverse with E_L and O (measuring, the FP64 refresh, the adjoint
// of ln|Psi|), and ln|Psi| alone.
//
// A = F[occ, occ] is antisymmetric, so only its upper triangle is kept, packed
// by rows (r <-> i < j), and every step of an elimination takes a pair of
// indices (p, q) at once: with a = A_pq, c_i = A_ip / a and d_i = A_iq,
//   A_ij += d_i c_j - c_i d_j                   (i, j not p, q).
// Gauss-Jordan over N/2 such steps, with
//   A_pj = d_j / a,  A_qj = -c_j,  A_pq = -1/a  afterwards,
// leaves A^{-1} in place, without any permutation (block pivots of an
// antisymmetric matrix; p is the next index, q the largest entry of its row,
// Bunch's partial pivoting).  That is N^3 / 2 multiply-adds against N^3 of a
// general inverse.  ln|Pf A| = sum of ln|a| needs the steps on the rows that are
// left only (Parlett and Reid), N^3 / 6.
//
// What bounds it: the FP64 pipe, which takes one warp FMA per 16 cycles per SM
// whatever the active lanes; so lanes run over the packed triangle (49 full
// rounds at 56 electrons, not 56 rows of two half-empty ones), pairs (i, j) come
// from a table, and 16 warps per SM hide the rest: it is 84 to 87 % busy.  16,384
// samples at 56 electrons: inverse, E_L and O 4.1 ms (10.3 ms with the general
// inverse of the walkers), the adjoint 3.6 ms (8.6), ln|Psi| 1.5 ms (5.7).
#include "ansatz.cuh"
#include "common.cuh"
#include "kernels.h"

namespace vmc {

namespace {

// packed index of i < j
__device__ __forceinline__ int tri(int N, int i, int j) { return i * (2 * N - i - 1) / 2 + j - i - 1; }

// A_ij of the packed triangle, i != j
__device__ __forceinline__ double get(const double* A, int N, int i, int j) {
    return i < j ? A[tri(N, i, j)] : -A[tri(N, j, i)];
}
__device__ __forceinline__ void put(double* A, int N, int i, int j, double v) {
    if (i < j) A[tri(N, i, j)] = v;
    else A[tri(N, j, i)] = -v;
}

// column of the warp's largest magnitude (to the upper 32 bits) among its lanes'
// two candidates; -1 if all vanish or one is not finite
__device__ __forceinline__ int pivot(double v0, int j0, double v1, int j1) {
    const uint32_t h0 = (uint32_t)__double2hiint(v0) & 0x7fffffffu, h1 = (uint32_t)__double2hiint(v1) & 0x7fffffffu;
    const uint32_t m = __reduce_max_sync(VMC_FULL_MASK, max(h0, h1));
    if (m >= 0x7ff00000u) return -1;
    const bool t0 = h0 == m && v0 != 0.0, t1 = h1 == m && v1 != 0.0;
    const uint32_t b = __ballot_sync(VMC_FULL_MASK, t0 || t1);
    if (b == 0u) return -1;
    return __shfl_sync(VMC_FULL_MASK, t0 ? j0 : j1, __ffs(b) - 1);
}

// A <- A^{-1} in place; cd: N pairs of scratch.  False if singular.
__device__ bool invert_packed(double* A, double2* cd, const uint16_t* ij, int N, int P) {
    const int lane = threadIdx.x & 31;
    uint64_t left = N == 64 ? ~0ull : (1ull << N) - 1ull;
    while (left) {
        const int p = __ffsll((long long)left) - 1;
        left &= left - 1;
        const int j1 = lane + 32;
        const bool l0 = (left >> lane) & 1ull, l1 = (left >> j1) & 1ull;
        const int q = pivot(l0 ? get(A, N, p, lane) : 0.0, lane, l1 ? get(A, N, p, j1) : 0.0, j1);
        if (q < 0) return false;
        left &= ~(1ull << q);
        const double ai = 1.0 / get(A, N, p, q);
        double2 v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            v[h] = make_double2(0.0, 0.0);
            if (i < N && i != p && i != q) v[h] = make_double2(get(A, N, i, p) * ai, get(A, N, i, q));
            if (i < N) cd[i] = v[h];
        }
        __syncwarp();
#pragma unroll 4
        for (int r = lane; r < P; r += 32) {
            const int t = ij[r];
            const double2 x = cd[t & 255], y = cd[t >> 8];
            A[r] = fma(x.y, y.x, fma(-x.x, y.y, A[r]));   // rows p and q meet zeros
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            if (i < N && i != p && i != q) {
                put(A, N, p, i, v[h].y * ai);
                put(A, N, q, i, -v[h].x);
            }
        }
        if (lane == 0) put(A, N, p, q, -ai);
        __syncwarp();
    }
    return true;
}

// ln|Pf A|; A is overwritten.  -infinity if a pivot row vanishes.
__device__ double log_pfaffian(double* A, double2* cd, const uint16_t* ij, int N, int P) {
    const int lane = threadIdx.x & 31;
    double mine = 1.0;   // lane k / 2 keeps step k's pivot: one logarithm for all at the end
    for (int k = 0; k < N; k += 2) {
        const int ja = lane + k + 1, jb = ja + 32;
        const int rk = tri(N, k, k + 1) - k - 1;   // row k: A[rk + j]
        const int q = pivot(ja < N ? A[rk + ja] : 0.0, ja, jb < N ? A[rk + jb] : 0.0, jb);
        if (q < 0) return -INFINITY;
        const int m = k + 1;
        if (q != m) {   // exchange indices m and q
            for (int i = k + lane; i < N; i += 32) {
                if (i == m || i == q) continue;
                const double x = get(A, N, i, m), y = get(A, N, i, q);
                put(A, N, i, m, y);
                put(A, N, i, q, x);
            }
            __syncwarp();
            if (lane == 0) A[tri(N, m, q)] = -A[tri(N, m, q)];
            __syncwarp();
        }
        const double a = A[rk + m];
        if (lane == k >> 1) mine = a;
        const double ai = 1.0 / a;
        for (int i = k + 2 + lane; i < N; i += 32)
            cd[i] = make_double2(-A[rk + i] * ai, -A[tri(N, m, i)]);   // (A_ip / a, A_iq)
        __syncwarp();
#pragma unroll 4
        for (int r = (k + 2 < N ? tri(N, k + 2, k + 3) : P) + lane; r < P; r += 32) {
            const int t = ij[r];
            const double2 x = cd[t & 255], y = cd[t >> 8];
            A[r] = fma(x.y, y.x, fma(-x.x, y.y, A[r]));
        }
        __syncwarp();
    }
    return warp_sum(log(fabs(mine)));
}

__device__ __forceinline__ void fill_pairs(uint16_t* ij, const uint32_t* fulltab, int P) {
    for (int r = threadIdx.x; r < P; r += blockDim.x) {
        const uint32_t f = fulltab[r];
        ij[r] = (uint16_t)(((f >> 16) & 255u) | (f >> 24) << 8);
    }
}

}  // namespace

// shared memory: the pair table, then per warp the triangle, the scratch pairs,
// the correlator states and the occupation
// (the scratch pairs also hold a queue of 32 words)
__host__ __device__ inline int scratch_pairs(int N) { return N < 8 ? 8 : N; }
__host__ __device__ inline size_t warp_bytes64(int N, int P, int ncorr) {
    return ((size_t)P * 8 + 8 + (size_t)scratch_pairs(N) * 16 + (size_t)ncorr * 4 + 64 + 15) / 16 * 16;
}
size_t measure64_smem(int N, int P, int ncorr, int warps) {
    return ((size_t)P * 2 + 15) / 16 * 16 + warps * warp_bytes64(N, P, ncorr);
}

__global__ void __launch_bounds__(128) k_measure64(SampleArgs a, const uint32_t* fulltab) {
    extern __shared__ __align__(16) unsigned char smem[];
    const DevProblem& pb = a.pb;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int N = pb.N, P = pb.P, ns = pb.ns, nu = pb.nu;
    uint16_t* ij = (uint16_t*)smem;
    fill_pairs(ij, fulltab, P);
    __syncthreads();
    unsigned char* base = smem + ((size_t)P * 2 + 15) / 16 * 16 + wid * warp_bytes64(N, P, pb.ncorr);
    double2* cd = (double2*)base;
    double* A = (double*)(cd + scratch_pairs(N));
    uint32_t* cidx = (uint32_t*)(A + P + (P & 1));
    uint8_t* occ = (uint8_t*)(cidx + pb.ncorr);
    const int64_t t0 = (int64_t)blockIdx.x * (blockDim.x >> 5) + wid;
    if (t0 >= a.n_walkers) return;
    const int64_t s = a.w0 + t0;

    // ---- the configuration --------------------------------------------------
    uint64_t up = 0, dn = 0;
    bool bad = false;
    for (int i = lane; i < N; i += 32) {
        const int o = a.walker_occ[s * N + i];
        occ[i] = (uint8_t)o;
        if (o >= pb.M) bad = true;
        else if (o < ns) up |= 1ull << o;
        else dn |= 1ull << (o - ns);
        if (i > 0 && a.walker_occ[s * N + i - 1] >= o) bad = true;
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
    for (int r = lane; r < P; r += 32) A[r] = __ldg(pb.F64 + occ[ij[r] & 255] * pb.M + occ[ij[r] >> 8]);
    for (int c = lane; c < pb.ncorr; c += 32) {
        uint32_t idx = 0, wgt = 1;
        for (int j = pb.corr_ptr[c]; j < pb.corr_ptr[c + 1]; ++j) {
            const int t = pb.corr_sites[j];
            idx += wgt * (uint32_t)(((up >> t) & 1ull) + 2ull * ((dn >> t) & 1ull));
            wgt <<= 2;
        }
        cidx[c] = idx;
    }
    __syncwarp();
    if (!invert_packed(A, cd, ij, N, P)) {
        if (lane == 0) atomicOr(a.status, ST_SINGULAR);
        return;
    }

    // ---- local energy (Hubbard): a lane per open hop ------------------------
    if (a.want_energy && pb.ham == 0) {
        double e = 0.0;
        // hops i -> neighbour k of its site, queued as (electron, neighbour entry)
        // until 32 are there; the queue lies in the scratch pairs
        uint32_t* queue = (uint32_t*)cd;
        int nq = 0;
        auto hop = [&](uint32_t en) {
            const int i = (int)(en & 255u), k = (int)(en >> 8), p = occ[i], spin = p >= ns;
            const int q = spin * ns + pb.nbr_site[k];
            // sum_{j != i} F[q][o_j] X_ij, F[q][o] = -F[o][q]
            double d = 0.0;
            int below = i - 1;   // packed index of (j, i), j < i: advances by N - j - 2
            const int above = tri(N, i, i + 1) - i - 1;
#pragma unroll 4
            for (int j = 0; j < N; ++j) {
                const double x = j < i ? -A[below] : j > i ? A[above + j] : 0.0;
                below += N - j - 2;
                d = fma(-__ldg(pb.F64 + occ[j] * pb.M + q), x, d);
            }
            // the correlators' part
            const int sp = p - spin * ns, sq = q - spin * ns;
            const int total = (pb.site_cptr[sp + 1] - pb.site_cptr[sp]) + (pb.site_cptr[sq + 1] - pb.site_cptr[sq]);
            double rc = 1.0;
            for (int t = 0; t < total; ++t) {
                int c;
                const int newi = corr_entry(pb, cidx, sp, sq, spin + 1, t, &c);
                if (c >= 0) rc *= __ldg(pb.C64 + pb.corr_off[c] + newi) * __ldg(pb.iC64 + pb.corr_off[c] + cidx[c]);
            }
            e += pb.nbr_t[k] * (d * rc);   // -t (Pf ratio = -d) rc
        };
        for (int i = 0; i < N; ++i) {
            const int p = occ[i], spin = p >= ns, sp = p - spin * ns;
            const uint64_t m = spin ? dn : up;
            const int k1 = pb.nbr_ptr[sp + 1];
            for (int k0 = pb.nbr_ptr[sp]; k0 < k1; k0 += 32) {
                const int k = k0 + lane;
                const bool open = k < k1 && !((m >> pb.nbr_site[k < k1 ? k : k0]) & 1ull);
                const uint32_t b = __ballot_sync(VMC_FULL_MASK, open);
                const int at = nq + __popc(b & ((1u << lane) - 1u));
                // a full group goes at once; the queue never holds more than 32
                uint32_t mine = 0;
                if (open) {
                    if (at < 32) queue[at] = (uint32_t)i | (uint32_t)k << 8;
                    else mine = (uint32_t)i | (uint32_t)k << 8;
                }
                nq += __popc(b);
                if (nq >= 32) {
                    __syncwarp();
                    const uint32_t en = queue[lane];
                    __syncwarp();
                    if (open && at >= 32) queue[at - 32] = mine;
                    nq -= 32;
                    hop(en);
                }
            }
        }
        __syncwarp();
        if (lane < nq) hop(queue[lane]);
        e = warp_sum(e) + pb.U * (double)__popcll(up & dn);
        if (!isfinite(e) && lane == 0) atomicOr(a.status, ST_NONFINITE);
        if (a.s_E && lane == 0) a.s_E[s] = e;
    }

    // ---- derivative ratios ----------------------------------------------------
    if (a.bgrad) {
        // adjoint: grad += w_s O(n_s)
        const double ws = a.bw[s];
        for (int c = lane; c < pb.ncorr; c += 32) {
            const int64_t k = pb.corr_off[c] + cidx[c];
            atomicAdd(a.bgrad + k, ws / pb.C64[k]);
        }
        for (int r = lane; r < P; r += 32) {
            const int t = ij[r];
            atomicAdd(a.bgrad + pb.ncp + pb.rowbase[occ[t & 255]] + occ[t >> 8], -(ws * A[r]));
        }
        return;
    }
    if (a.s_X) {   // the whole inverse, for the ab initio energy's pass
        double* dst = (double*)a.s_X + t0 * N * N;
        for (int t = lane; t < N * N; t += 32) dst[t] = t / N == t % N ? 0.0 : get(A, N, t / N, t % N);
        for (int i = lane; i < N; i += 32) a.s_pos[s * a.Nst + i] = occ[i];
    }
    for (int i = lane; i < N; i += 32)
        if (a.s_occ) a.s_occ[s * a.Nst + i] = occ[i];
    if (a.s_lnrun && lane == 0) a.s_lnrun[s] = 0.0;
    if (a.s_cidx)
        for (int c = lane; c < pb.ncorr; c += 32) a.s_cidx[s * a.ncst + c] = (cstate_t)cidx[c];
    for (int e = lane; e < P; e += 32) {
        const uint16_t t = pb.pairtab[e];
        const double w = -A[tri(N, t & 255, t >> 8)];   // (A^{-1})_ba
        if (a.s_pf64) a.s_pf64[s * a.Pst + e] = w;
        if (a.s_pf32) a.s_pf32[s * a.Pst + e] = (float)w;
        if (a.s_pf16) a.s_pf16[s * a.Pst + e] = __float2bfloat16_rn((float)w);
    }
}

// ln|Pf(F[occ, occ])| + sum_c ln|C_c| per stored sample
__global__ void __launch_bounds__(128) k_logpsi(LogPsiArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const DevProblem& pb = a.pb;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int N = pb.N, P = pb.P;
    uint16_t* ij = (uint16_t*)smem;
    fill_pairs(ij, a.fulltab, P);
    __syncthreads();
    unsigned char* base = smem + ((size_t)P * 2 + 15) / 16 * 16 + wid * warp_bytes64(N, P, 0);
    double2* cd = (double2*)base;
    double* A = (double*)(cd + scratch_pairs(N));
    const int64_t s = (int64_t)blockIdx.x * (blockDim.x >> 5) + wid;
    if (s >= a.n_s) return;
    const uint8_t* occ = a.s_occ + s * a.Nst;
    for (int r = lane; r < P; r += 32) A[r] = __ldg(pb.F64 + occ[ij[r] & 255] * pb.M + occ[ij[r] >> 8]);
    __syncwarp();
    const double lp = log_pfaffian(A, cd, ij, N, P);
    const cstate_t* ci = a.s_cidx + s * a.ncst;
    double lc = 0.0;
    for (int c = lane; c < pb.ncorr; c += 32) lc += log(fabs(pb.C64[pb.corr_off[c] + ci[c]]));
    lc = warp_sum(lc);
    if (lane == 0) a.out[s] = lp + lc;
}

}  // namespace vmc
