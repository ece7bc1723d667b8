// One-pass Eq. 7 product and gradient pass over the O store with FP64 sums
// (FP64 arithmetic; FP32 pairs for the FP32 store), without atomics.
//
// A CTA works through its samples in tiles.  Gather: a warp per sample forms
// t_s = O_s . V.  Scatter: t_s O_s is added to shared-memory images of the
// pairing block.  An image belongs to `owners` warps that split the samples'
// elements by their smaller orbital p = occ[a] (boundaries of about equal
// expected work), so two warps never touch one address, whatever samples they
// are at: an update is a plain load, add and store, and the only
// synchronisation is one barrier per tile between gather and scatter.  How many
// images and owners: plan_pass.  A warp without a part in the scatter gathers the
// next tile meanwhile.  The sums have a fixed order.  Small correlator blocks
// enter the images too (in FP64, a warp's lanes over the correlators); larger ones
// are summed from the t_s by a kernel of their own.
//
// What bounds it: the FP64 store's pass the FP64 pipe (two FMAs per element, 74 %
// busy), the FP32 store's issue slots and shared-memory latency (32 warps).  8x8
// lattice, 28 + 28 electrons: FP64 store, 65,536 samples 594 us (825 us with FP64
// shared atomics), FP32 store, 131,072 samples 919 us (1,299 us with two shared
// FP32 atomics per element).  At an earlier state (600 / 930 us), warps per CTA: 16
// 695 / 1,225 us; the FP32 store's gather in FP64 1,470 us (conversions fill the FP64
// pipe); scatter rounds of 4 elements per lane, skipped by the whole warp, 643 / 976
// us.  Few electrons are bound by the latency of a tile's phases.
//
// Elements go in the row-major order of electron pairs a < b (fulltab), in
// which an owner's share of a sample is one stretch; the tile's occupations
// and row bases sit in shared memory.  The second read of the values comes out
// of L2.
//
// FP32 pairs: the FP64 pipe of this GPU retires one warp FMA per 16 cycles per
// SM, so the FP32 store's passes stay off it.  The v table holds
// each FP64 value as an FP32 pair (hi, lo); a product w v = w hi + w lo is
// split exactly into its rounded value and the FMA error term; the per-lane
// sums and the images are FP32 pairs kept by Knuth's two-sum.  The rounded
// intrinsics keep the compiler from fusing the error arithmetic.
#include <type_traits>
#include "common.cuh"
#include "kernels.h"

namespace vmc {

namespace {

__device__ __forceinline__ void ff_add(float& sh, float& sl, float p, float err) {
    const float s = __fadd_rn(sh, p);
    const float bp = __fsub_rn(s, sh);
    const float e = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bp)), __fsub_rn(p, bp));
    sh = s;
    sl = __fadd_rn(sl, __fadd_rn(e, err));
}

__device__ __forceinline__ float2 ff_split(double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}

__device__ __forceinline__ float load_w(const float* p) { return __ldg(p); }
__device__ __forceinline__ double load_w(const double* p) { return __ldg(p); }
__device__ __forceinline__ float load_w(const __nv_bfloat16* p) {
    return __uint_as_float((uint32_t)__ldg((const unsigned short*)p) << 16);
}
// FP32 to FP64 by its bits (a conversion would take the FP64 pipe's time again)
__device__ __forceinline__ double widen(double w) { return w; }
__device__ __forceinline__ double widen(float w) {
    const uint32_t u = __float_as_uint(w), m = u & 0x7fffffffu;
    double d = __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
    if (__any_sync(__activemask(), m - 0x00800000u >= 0x7f000000u)) d = (double)w;   // not a normal number in some lane
    return d;
}

// Element arithmetic: plain FP64, or FP32 pairs for the FP32 store.
struct PlainAcc {
    using Elem = double;   // a table or image entry
    static __device__ __forceinline__ Elem make(double v) { return v; }
    static __device__ __forceinline__ double value(Elem v) { return v; }
    static __device__ __forceinline__ void sum(Elem& s, Elem v) { s += v; }
    template <typename W> static __device__ __forceinline__ void add(Elem& s, W w, Elem v) { s = fma(widen(w), v, s); }
};
struct PairAcc {
    using Elem = float2;
    static __device__ __forceinline__ Elem make(double v) { return ff_split(v); }
    static __device__ __forceinline__ double value(Elem v) { return (double)v.x + (double)v.y; }
    static __device__ __forceinline__ void sum(Elem& s, Elem v) { ff_add(s.x, s.y, v.x, v.y); }
    static __device__ __forceinline__ void add(Elem& s, float w, Elem v) {
        const float p = __fmul_rn(w, v.x);
        ff_add(s.x, s.y, p, fmaf(w, v.y, fmaf(w, v.x, -p)));
    }
};

// Sums of K values over the warp, the k-th in the lanes from 32 k / K on: the first
// log2 K steps halve the values that a lane carries on, so four sums are 6 FP64 adds
// (16 cycles each, whatever the lanes do), not 20.
template <int K>
__device__ __forceinline__ double warp_sums(double (&v)[K]) {
    int o = 16;
#pragma unroll
    for (int n = K; n > 1; n /= 2, o /= 2) {
        const bool up = threadIdx.x & o;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
            const double give = up ? v[i] : v[i + n / 2], keep = up ? v[i + n / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(VMC_FULL_MASK, give, o);
        }
    }
#pragma unroll
    for (; o > 0; o /= 2) v[0] += __shfl_xor_sync(VMC_FULL_MASK, v[0], o);
    return v[0];
}

constexpr int kU = 4, kUs = 2;   // elements per lane in flight, gather and scatter

// shared memory of one tile buffer
template <typename E, int K, int NW>
struct TileBuf {
    E t[kPassTile][K];
    int16_t rb[kPassTile][64];               // row bases of the occupied orbitals
    uint8_t occ[kPassTile][64];
    uint16_t start[kPassTile][NW + 1];   // first element (rank) of each owner
};

template <typename ST, int K, bool GATHER, int NW>
__device__ void pass_run(const PassArgs& a, int cta, int ncta, unsigned char* smem) {
    using A = typename std::conditional<std::is_same<ST, float>::value, PairAcc, PlainAcc>::type;
    using E = typename A::Elem;
    const DevProblem& pb = a.pb;
    const int npf = pb.npf, N = pb.N, P = pb.P, ni = a.ni, owners = a.owners, nimg = a.nimg;
    E* img = (E*)smem;                                           // [ni][nimg][K]
    E* vpf = img + (size_t)ni * nimg * K;                        // [npf][K]
    TileBuf<E, K, NW>* buf = (TileBuf<E, K, NW>*)(vpf + (GATHER ? (size_t)npf * K : 0));   // [2]
    uint32_t* ft = (uint32_t*)(buf + 2);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < ni * nimg * K; i += blockDim.x) img[i] = E{};
    if (GATHER)
        for (int i = threadIdx.x; i < npf; i += blockDim.x)
#pragma unroll
            for (int kk = 0; kk < K; ++kk) vpf[i * K + kk] = A::make(a.V[kk * pb.nv + pb.ncp + i]);
    for (int i = threadIdx.x; i < P; i += blockDim.x) ft[i] = a.fulltab[i];
    // on the side: this CTA's share of Obar . V and of clearing the correlator sums
    if (GATHER && a.Obar) {
        double* red = (double*)buf;   // [K][NW]
        const int64_t per = (pb.nv + ncta - 1) / ncta, i1 = min(pb.nv, (cta + 1) * per);
        double d[K] = {};
        for (int64_t i = cta * per + threadIdx.x; i < i1; i += blockDim.x) {
            const double o = a.Obar[i];
#pragma unroll
            for (int kk = 0; kk < K; ++kk) d[kk] += o * a.V[kk * pb.nv + i];
        }
#pragma unroll
        for (int kk = 0; kk < K; ++kk) {
            d[kk] = warp_sum(d[kk]);
            if (lane == 0) red[kk * NW + wid] = d[kk];
        }
        __syncthreads();
        if (threadIdx.x < K) {
            double x = 0.0;
            for (int w = 0; w < NW; ++w) x += red[threadIdx.x * NW + w];
            a.obv_part[cta * K + threadIdx.x] = x;
        }
    }
    if (a.clear)
        for (int64_t i = (int64_t)cta * blockDim.x + threadIdx.x; i < a.nclear; i += (int64_t)ncta * blockDim.x)
            a.clear[i] = 0.0;
    __syncthreads();
    const ST* pf = (const ST*)a.s_pf;
    const int im = wid / owners, own = wid % owners;
    E* my = img + (size_t)im * nimg * K;   // (im >= ni: no part in the scatter)
    const int64_t per = (a.n_s + ncta - 1) / ncta;
    const int64_t s0 = min(a.n_s, cta * per), s1 = min(a.n_s, s0 + per);
    uint32_t below[4];   // the orbitals below the first one of owner `lane`, 32 to a word
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int b = a.bounds[min(lane, owners)] - 32 * k;
        below[k] = b >= 32 ? ~0u : b <= 0 ? 0u : (1u << b) - 1u;
    }
    int cur = 0;
    for (int64_t sb = s0; sb < s1; sb += kPassTile, cur ^= 1) {
        TileBuf<E, K, NW>& B = buf[cur];
        const int n = (int)min((int64_t)kPassTile, s1 - sb);
        // ---- gather: the warp's samples of the tile ------------------------
        for (int j = wid; j < n; j += NW) {
            const int64_t s = sb + j;
            int o[2], ck[2];
            double ic[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = lane + 32 * h;
                if (GATHER) ck[h] = i < pb.ncorr ? (int)(pb.corr_off[i] + a.s_cidx[s * a.ncst + i]) : -1;
                o[h] = i < N ? a.s_occ[s * a.Nst + i] : 255;
                if (i < N) {
                    B.occ[j][i] = (uint8_t)o[h];
                    B.rb[j][i] = (int16_t)pf_row_base(pb.M, o[h]);
                }
            }
            if (GATHER)
#pragma unroll
                for (int h = 0; h < 2; ++h) ic[h] = ck[h] >= 0 ? a.invC[ck[h]] : 0.0;
            int a0 = 0;   // electrons below the first orbital of owner `lane`
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t m = ((o[0] >> 5) == k ? 1u << (o[0] & 31) : 0u) | ((o[1] >> 5) == k ? 1u << (o[1] & 31) : 0u);
                a0 += __popc(__reduce_or_sync(VMC_FULL_MASK, m) & below[k]);
            }
            if (lane < owners) B.start[j][lane] = (uint16_t)(a0 * (2 * N - a0 - 1) / 2);
            if (lane == 0) B.start[j][owners] = (uint16_t)P;
            __syncwarp();
            if (GATHER) {
                E sum[K];
                double tc[K];
#pragma unroll
                for (int kk = 0; kk < K; ++kk) {
                    sum[kk] = A::make(0.0);
                    tc[kk] = 0.0;
                }
                for (int c = lane + 64; c < pb.ncorr; c += 32) {
                    const int64_t k = pb.corr_off[c] + a.s_cidx[s * a.ncst + c];
                    const double ic = a.invC[k];
#pragma unroll
                    for (int kk = 0; kk < K; ++kk) tc[kk] += a.V[kk * pb.nv + k] * ic;
                }
                double cv[2][K];   // the first two correlators of the lane: loaded before the row, used after it
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int kk = 0; kk < K; ++kk) cv[h][kk] = ck[h] >= 0 ? a.V[kk * pb.nv + ck[h]] : 0.0;
                const ST* row = pf + s * a.Pst;
                for (int r0 = lane; r0 < P; r0 += 32 * kU) {
                    decltype(load_w(row)) w[kU];
                    int pq[kU];
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const uint32_t f = ft[min(r0 + 32 * u, P - 1)];
                        w[u] = load_w(row + (f & 0xFFFFu));
                        pq[u] = B.rb[j][(f >> 16) & 255] + B.occ[j][f >> 24];
                    }
#pragma unroll
                    for (int u = 0; u < kU; ++u)
                        if (r0 + 32 * u < P)
#pragma unroll
                            for (int kk = 0; kk < K; ++kk) A::add(sum[kk], w[u], vpf[pq[u] * K + kk]);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int kk = 0; kk < K; ++kk) tc[kk] += cv[h][kk] * ic[h];
#pragma unroll
                for (int kk = 0; kk < K; ++kk) tc[kk] += A::value(sum[kk]);
                const double t = warp_sums<K>(tc);
                if ((lane & (32 / K - 1)) == 0) {
                    const int kk = lane / (32 / K);
                    a.T[s * a.ts + kk] = t;
                    B.t[j][kk] = A::make(t);
                }
            } else if (lane < K) {
                B.t[j][lane] = A::make(a.T[s * a.ts + lane]);
            }
        }
        __syncthreads();
        // ---- scatter: the owner's share of the image's samples ---------------
        for (int j = im < ni ? im : n; j < n; j += ni) {
            const ST* row = pf + (sb + j) * a.Pst;
            E t[K];
#pragma unroll
            for (int kk = 0; kk < K; ++kk) t[kk] = B.t[j][kk];
            const int r1 = B.start[j][own + 1];
            for (int r0 = B.start[j][own] + lane; r0 < r1; r0 += 32 * kUs) {
                decltype(load_w(row)) w[kUs];
                int pq[kUs];
#pragma unroll
                for (int u = 0; u < kUs; ++u) {
                    const uint32_t f = ft[min(r0 + 32 * u, P - 1)];
                    w[u] = load_w(row + (f & 0xFFFFu));
                    pq[u] = B.rb[j][(f >> 16) & 255] + B.occ[j][f >> 24];
                }
                E x[kUs][K];   // a sample's elements are at distinct addresses: loads first
#pragma unroll
                for (int u = 0; u < kUs; ++u)
#pragma unroll
                    for (int kk = 0; kk < K; ++kk) x[u][kk] = my[pq[u] * K + kk];
#pragma unroll
                for (int u = 0; u < kUs; ++u)
                    if (r0 + 32 * u < r1)
#pragma unroll
                        for (int kk = 0; kk < K; ++kk) {
                            A::add(x[u][kk], w[u], t[kk]);
                            my[pq[u] * K + kk] = x[u][kk];
                        }
            }
            if (nimg > npf)   // the correlators' part in FP64 (1 / C enters at the end): a block each, so no two meet
                for (int c = own * 32 + lane; c < pb.ncorr; c += 32 * owners) {
                    double* y = (double*)(my + (npf + pb.corr_off[c] + a.s_cidx[(sb + j) * a.ncst + c]) * K);
#pragma unroll
                    for (int kk = 0; kk < K; ++kk) y[kk] += a.T[(sb + j) * a.ts + kk];
                }
            __syncwarp();   // the next sample's elements may meet these addresses in other lanes
        }
    }
    __syncthreads();
    double* dst = a.pf_partial + (size_t)cta * nimg * K;
    for (int i = threadIdx.x; i < npf * K; i += blockDim.x) {
        E x = img[i];
        for (int k = 1; k < ni; ++k) A::sum(x, img[(size_t)k * nimg * K + i]);
        dst[i] = A::value(x);
    }
    for (int i = npf * K + threadIdx.x; i < nimg * K; i += blockDim.x) {
        double x = 0.0;
        for (int k = 0; k < ni; ++k) x += ((double*)img)[(size_t)k * nimg * K + i];
        dst[i] = x;
    }
}

// The CTAs' images added up, and what follows: out = raw / n - Obar (Obar . V)
// + shift V with partial out . V, or (GRAD) the means and the gradient.  Blocks
// [0, ceil(nimg / 32)) take 32 image entries each, 8 slices of the images; the
// other blocks the correlator sums that another kernel left in corr_raw.
// A small product is its launches: with Obar . V, the clearing and the correlators
// in the pass and everything after it here, 4x4 lattice, 4,096 samples, one vector
// went from five kernels and a memset at 75 us a call to two at 46.
template <int K, bool GRAD>
__global__ void __launch_bounds__(256) k_sr_finish(FinishArgs a) {
    if (a.stop && *a.stop) return;
    __shared__ double red[8][K][33];
    __shared__ double lead[K];   // Obar . V, or <E_L>
    const DevProblem& pb = a.pb;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w == 0) {
#pragma unroll
        for (int kk = 0; kk < (GRAD ? 1 : K); ++kk) {
            const double x = warp_sum_partials(a.lead_part, a.n_lead, kk, GRAD ? 1 : K);
            if (lane == 0) lead[kk] = GRAD ? x * a.inv_n : x;
        }
    }
    const int nb1 = (a.nimg + 31) / 32;
    double dot[K] = {};
    auto finish = [&](int64_t k, double* raw) {   // parameter k, its sums
#pragma unroll
        for (int kk = 0; kk < K; ++kk) raw[kk] = (k < pb.ncp ? raw[kk] * a.invC[k] : raw[kk]) * a.inv_n;
        if (GRAD) {
            a.Obar_out[k] = raw[0];
            a.Obar32_out[k] = (float)raw[0];
            a.g_out[k] = raw[1] - lead[0] * raw[0];
        } else {
            const double ob = a.Obar[k];
#pragma unroll
            for (int kk = 0; kk < K; ++kk) {
                const double v = a.V[kk * pb.nv + k], o = raw[kk] - ob * lead[kk] + a.shift * v;
                a.out[kk * pb.nv + k] = o;
                dot[kk] += o * v;
            }
        }
    };
    if ((int)blockIdx.x < nb1) {
        const int i = blockIdx.x * 32 + lane;
        double s[K] = {};
        if (i < a.nimg)
            for (int b0 = w; b0 < a.nblk; b0 += 64) {   // eight images in flight per thread
                double x[8][K];
#pragma unroll
                for (int u = 0; u < 8; ++u)
#pragma unroll
                    for (int kk = 0; kk < K; ++kk)
                        x[u][kk] = b0 + 8 * u < a.nblk ? a.part[((int64_t)(b0 + 8 * u) * a.nimg + i) * K + kk] : 0.0;
#pragma unroll
                for (int u = 0; u < 8; ++u)
#pragma unroll
                    for (int kk = 0; kk < K; ++kk) s[kk] += x[u][kk];
            }
#pragma unroll
        for (int kk = 0; kk < K; ++kk) red[w][kk][lane] = s[kk];
        __syncthreads();
        if (w == 0 && i < a.nimg) {
            double raw[K];
#pragma unroll
            for (int kk = 0; kk < K; ++kk) {
                raw[kk] = 0.0;
#pragma unroll
                for (int j = 0; j < 8; ++j) raw[kk] += red[j][kk][lane];
            }
            finish(i < pb.npf ? pb.ncp + i : i - pb.npf, raw);
        }
    } else {
        __syncthreads();
        const int64_t stride = (int64_t)(gridDim.x - nb1) * blockDim.x;
        for (int64_t k = (int64_t)(blockIdx.x - nb1) * blockDim.x + threadIdx.x; k < pb.ncp; k += stride) {
            double raw[K];
#pragma unroll
            for (int kk = 0; kk < K; ++kk) raw[kk] = a.corr_raw[k * a.cs + kk];
            finish(k, raw);
        }
    }
    if (!GRAD && a.dot_part) {
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < K; ++kk) {
            const double x = warp_sum(dot[kk]);
            if (lane == 0) red[w][kk][0] = x;
        }
        __syncthreads();
        if (threadIdx.x < K) {
            double x = 0.0;
            for (int j = 0; j < 8; ++j) x += red[j][threadIdx.x][0];
            a.dot_part[blockIdx.x * K + threadIdx.x] = x;
        }
    }
}

template <typename ST, int K, bool GATHER>
__global__ void __launch_bounds__(32 * pass_warps(K), 1) k_sr_pass(PassArgs a) {
    if (a.stop && *a.stop) return;
    extern __shared__ __align__(16) unsigned char smem[];
    pass_run<ST, K, GATHER, pass_warps(K)>(a, blockIdx.x, gridDim.x, smem);
}

// Several problems in one launch: CTAs [cta0[b], cta0[b + 1]) serve problem
// b, each with the shared-memory layout of its own problem.
template <typename ST>
__global__ void __launch_bounds__(32 * pass_warps(1), 1) k_sr_pass_batch(const PassArgs* __restrict__ args,
                                                                         const int* __restrict__ cta0, int n) {
    extern __shared__ __align__(16) unsigned char smem[];
    int b = 0;
    while (b + 1 < n && (int)blockIdx.x >= cta0[b + 1]) ++b;
    if ((int)blockIdx.x >= cta0[n]) return;
    pass_run<ST, 1, true, pass_warps(1)>(args[b], blockIdx.x - cta0[b], cta0[b + 1] - cta0[b], smem);
}

template <typename ST, int K, bool GATHER>
cudaError_t launch(const PassArgs& a, int grid, size_t smem, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_sr_pass<ST, K, GATHER>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_sr_pass<ST, K, GATHER><<<grid, 32 * pass_warps(K), smem, st>>>(a);
    return cudaGetLastError();
}

template <typename ST>
cudaError_t launch_k(const PassArgs& a, int K, bool gather, int grid, size_t smem, cudaStream_t st) {
    if (!gather) return launch<ST, 2, false>(a, grid, smem, st);
    if (K == 1) return launch<ST, 1, true>(a, grid, smem, st);
    if (K == 2) return launch<ST, 2, true>(a, grid, smem, st);
    return launch<ST, 4, true>(a, grid, smem, st);
}

}  // namespace

// shared memory with ni images (a table or image entry is 8 bytes in either arithmetic)
size_t pass_smem(int npf, int nimg, int P, int K, bool gather, int ni) {
    const size_t tile = K == 1   ? sizeof(TileBuf<double, 1, pass_warps(1)>)
                        : K == 2 ? sizeof(TileBuf<double, 2, pass_warps(2)>)
                                 : sizeof(TileBuf<double, 4, pass_warps(4)>);
    return ((size_t)nimg * ni + (gather ? npf : 0)) * K * 8 + 2 * tile + (size_t)P * 4;
}

cudaError_t launch_sr_pass(int store_bytes, const PassArgs& a, int K, bool gather, int grid, size_t smem, cudaStream_t st) {
    if (store_bytes == 8) return launch_k<double>(a, K, gather, grid, smem, st);
    if (store_bytes == 4) return launch_k<float>(a, K, gather, grid, smem, st);
    return launch<__nv_bfloat16, 2, false>(a, grid, smem, st);   // the BF16 store's means only
}

cudaError_t launch_sr_pass_batch(int store_bytes, int blocks, size_t smem, cudaStream_t st, const PassArgs* args,
                                 const int* cta0, int n) {
    auto kern = store_bytes == 8 ? k_sr_pass_batch<double> : k_sr_pass_batch<float>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<blocks, 32 * pass_warps(1), smem, st>>>(args, cta0, n);
    return cudaGetLastError();
}

cudaError_t launch_sr_finish(const FinishArgs& a, int K, bool grad, int grid, cudaStream_t st) {
    if (grad) k_sr_finish<2, true><<<grid, 256, 0, st>>>(a);
    else if (K == 1) k_sr_finish<1, false><<<grid, 256, 0, st>>>(a);
    else if (K == 2) k_sr_finish<2, false><<<grid, 256, 0, st>>>(a);
    else k_sr_finish<4, false><<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace vmc
