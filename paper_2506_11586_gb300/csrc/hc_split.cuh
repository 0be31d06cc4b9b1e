// hc_split.cuh -- transforms split over a cluster of 2^LOGP CTAs, for the latency of few
// polynomials: the parts of a kernel (used by hc_keyswitch.cuh too), and the forward
// transform, the inverse transform and the standalone product built from them.
//
// The first LOGP forward stages pair residues N / 2^LOGP apart.  Each CTA computes them in
// registers for its slice of the pairs and writes the results into the CTA that owns them
// (distributed shared memory); after a cluster barrier the remaining stages are local to
// the CTA (the engine's PART mode).  The inverse runs the other way round, N^-1 merged into
// the last stage.  The arithmetic is the one-CTA transform's, stage by stage.
// A transform of one limb by one CTA is bound by the latency of its warps (10 us at N = 8192,
// 19 at 16384, whatever the number of idle SMs); split, 4.5 and 9 us.  Where the split stops
// paying: split_units_ntt, split_units_product (hc_internal.h).
#pragma once

#include <atomic>

#include "hc_async.cuh"
#include "hc_ntt.cuh"

namespace hc {

// NG groups of T threads, NP polynomials at a time: group g takes the polynomials
// g*NP .., (g + NG)*NP ...  2^LOGC residues of each per thread.
//   latency (NG = 4, NP = 1): with few units in flight a CTA has an SM to itself, and the
//     time is the instructions of one warp times their latency, so the polynomials run
//     side by side.
//   throughput (NG = 1, NP = 2): one set of twiddle loads for two polynomials, more CTAs
//     per SM.
template <int LOGN_, int LOGP_, int NG_, int NP_, int LOGC_ = 3, int WARPS_ = 24>
struct SplitShape {
    static constexpr int LOGN = LOGN_, LOGP = LOGP_, CS = 1 << LOGP, NG = NG_, NP = NP_;
    template <int P>
    using CfgP = NttCfg<LOGN - LOGP, LOGC_, P, 1, NG>;
    using Cfg = CfgP<1>;
    static constexpr int NL = Cfg::N, T = Cfg::T, C = Cfg::C, ITEMS = C / CS, THREADS = T * NG;
    // registers for WARPS warps per SM
    static constexpr int MINB = THREADS * 2 > 32 * WARPS_ ? 1 : 32 * WARPS_ / THREADS;
    static_assert(ITEMS >= 1 && NL / CS == ITEMS * T, "whole slices of the cross stages");
};

// first LOGP stages of NP polynomials (src, pstride apart) for this thread's slice, results
// into their owners' buffers at sm + off, NL apart.  slice: the thread's first pair.
template <class S, int NP, bool SP>
__device__ __forceinline__ void split_fwd_cross(const uint64_t *src, size_t pstride, const uint64_t *sm, uint32_t off,
                                                uint32_t slice, const LimbConst &lc, const TwArith<SP> &ar)
{
    constexpr int CS = S::CS, ITEMS = S::ITEMS, T = S::T, NL = S::NL;
    uint64_t v[NP][ITEMS][CS];
    const uint64_t *a = src + slice;
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int it = 0; it < ITEMS; ++it)
#pragma unroll
            for (int c = 0; c < CS; ++c) v[p][it][c] = ld_data(a + p * pstride + it * T + c * NL);
    static_for<0, S::LOGP>([&](auto sc) {
        constexpr int s = decltype(sc)::value, half = CS >> (s + 1);
#pragma unroll
        for (int lam = 0; lam < (1 << s); ++lam) {
            const ulonglong2 w = __ldg(lc.tw_f + (1 << s) + lam);
#pragma unroll
            for (int jj = 0; jj < half; ++jj) {
                const int k = lam * 2 * half + jj;
#pragma unroll
                for (int p = 0; p < NP; ++p)
#pragma unroll
                    for (int it = 0; it < ITEMS; ++it) {
                        const uint64_t X = v[p][it][k], t = ar.mul(v[p][it][k + half], w);
                        v[p][it][k] = X + t;
                        v[p][it][k + half] = ar.sub(X, t);
                    }
            }
        }
    });
#pragma unroll
    for (int c = 0; c < CS; ++c) {
        const uint32_t to = cluster_map(sm, c) + (off + slice) * 8;
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) st_cluster_u64(to + (p * NL + it * T) * 8, v[p][it][c]);
    }
}

// last LOGP stages of NP polynomials for this thread's slice, read from their owners'
// buffers at sm + off (natural order, lazy), canonical: v[p][it][c] is element
// slice + it*T + c*NL
template <class S, int NP, bool SP>
__device__ __forceinline__ void split_inv_cross(uint64_t (&v)[NP][S::ITEMS][S::CS], const uint64_t *sm, uint32_t off,
                                                uint32_t slice, const LimbConst &lc, const TwArith<SP> &ar)
{
    constexpr int LOGP = S::LOGP, CS = S::CS, ITEMS = S::ITEMS, T = S::T, NL = S::NL;
    if constexpr (SP) {  // inputs of the last stage: sums throughout, or a product in an earlier one
        constexpr uint64_t sums = inv_in_bound<typename S::Cfg, S::Cfg::NROUNDS, LOGP>() << (LOGP - 1);
        static_assert(sums <= kFoldStage && (kFoldMax << LOGP) <= kFoldStage, "cross stages overflow");
    }
    const ulonglong2 wn = make_ulonglong2(lc.ninv, lc.ninv_s), wnw = make_ulonglong2(lc.ninvw, lc.ninvw_s);
#pragma unroll
    for (int c = 0; c < CS; ++c) {
        const uint32_t from = cluster_map(sm, c) + (off + slice) * 8;
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) v[p][it][c] = ld_cluster_u64(from + (p * NL + it * T) * 8);
    }
    static_for<0, LOGP>([&](auto sc) {
        constexpr int s = decltype(sc)::value, dist = 1 << s, ngrp = CS >> (s + 1);
        const uint64_t qs = ar.q << (S::LOGN - LOGP + s);  // bound of the stage's inputs (Shoup)
#pragma unroll
        for (int g = 0; g < ngrp; ++g) {
            const ulonglong2 w = __ldg(lc.tw_i + ngrp + g);
#pragma unroll
            for (int jj = 0; jj < dist; ++jj) {
                const int k = g * 2 * dist + jj;
#pragma unroll
                for (int p = 0; p < NP; ++p)
#pragma unroll
                    for (int it = 0; it < ITEMS; ++it) {
                        const uint64_t X = v[p][it][k], Y = v[p][it][k + dist];
                        if constexpr (s == LOGP - 1) {
                            v[p][it][k] = ar.template div_canon<S::LOGN>(X + Y, wn);
                            v[p][it][k + dist] = ar.mul_canon(ar.sub(X, Y, qs), wnw);
                        } else {
                            v[p][it][k] = X + Y;
                            v[p][it][k + dist] = ar.mul(ar.sub(X, Y, qs), w);
                        }
                    }
            }
        }
    });
}

// unit u of a segment table (segment units: limb-major) -> source offset and constants
template <int NS>
__device__ __forceinline__ const NttSeg &split_unit(const NttSegsT<NS> &segs, uint32_t u, size_t n, size_t &off,
                                                    uint32_t &limb)
{
    uint32_t si = 0;
    while (si + 1 < segs.n && u >= segs.s[si + 1].cta_begin) ++si;
    const NttSeg &sg = segs.s[si];
    const uint32_t local = u - sg.cta_begin;
    limb = sg.limb0 + local / sg.n_groups;
    off = ((size_t)(local % sg.n_groups) * sg.L + limb) * n;
    return sg;
}

// forward NTT of one polynomial limb per cluster, canonical
template <class S, int NS, bool SP>
__global__ void __cluster_dims__(S::CS, 1, 1) __launch_bounds__(S::THREADS, S::MINB)
k_ntt_fwd_split(const __grid_constant__ NttSegsT<NS> segs)
{
    static_assert(S::NG == 1 && S::NP == 1, "one polynomial per cluster");
    using Cfg = typename S::Cfg;
    constexpr int C = S::C, T = S::T, NL = S::NL;
    extern __shared__ __align__(16) uint64_t sm[];  // [NL]
    const int tid = threadIdx.x;
    const uint32_t rank = cluster_rank();
    size_t off;
    uint32_t limb;
    const NttSeg &sg = split_unit(segs, blockIdx.x >> S::LOGP, (size_t)1 << S::LOGN, off, limb);
    const LimbConst &lc = sg.limbs[limb];
    const TwArith<SP> ar = tw_arith<SP>(lc);
    cluster_sync();  // every CTA of the cluster is running before one writes into another
    pdl_begin();
    split_fwd_cross<S, 1, SP>(after_wait(sg.in) + off, 0, sm, 0, rank * (NL / S::CS) + tid, lc, ar);
    cluster_sync();  // this CTA's part is complete, and every load of an in-place transform done
    uint64_t x[1][C];
#pragma unroll
    for (int r = 0; r < C; ++r) x[0][r] = sm[tid + r * T];
    fwd_rounds<Cfg, 0, S::LOGP, SP>(x, sm, lc.tw_f, nullptr, ar, tid, S::CS + (int)rank);
    ulonglong2 *d = reinterpret_cast<ulonglong2 *>(sg.out + off + rank * NL + tid * C);
#pragma unroll
    for (int r = 0; r < C; r += 2) d[r / 2] = make_ulonglong2(ar.canon(x[0][r]), ar.canon(x[0][r + 1]));
}

// inverse NTT of one polynomial limb per cluster
template <class S, int NS, bool SP>
__global__ void __cluster_dims__(S::CS, 1, 1) __launch_bounds__(S::THREADS, S::MINB)
k_ntt_inv_split(const __grid_constant__ NttSegsT<NS> segs)
{
    static_assert(S::NG == 1 && S::NP == 1, "one polynomial per cluster");
    using Cfg = typename S::Cfg;
    constexpr int C = S::C, T = S::T, NL = S::NL;
    extern __shared__ __align__(16) uint64_t sm[];  // [NL]
    const int tid = threadIdx.x;
    const uint32_t rank = cluster_rank();
    size_t off;
    uint32_t limb;
    const NttSeg &sg = split_unit(segs, blockIdx.x >> S::LOGP, (size_t)1 << S::LOGN, off, limb);
    const LimbConst &lc = sg.limbs[limb];
    const TwArith<SP> ar = tw_arith<SP>(lc);
    pdl_begin();
    const ulonglong2 *src = reinterpret_cast<const ulonglong2 *>(after_wait(sg.in + off + rank * NL + tid * C));
    uint64_t x[1][C];
#pragma unroll
    for (int r = 0; r < C; r += 2) {
        const ulonglong2 a = ld_data(src + r / 2);
        x[0][r] = a.x;
        x[0][r + 1] = a.y;
    }
    inv_transform<Cfg, S::LOGP>(x, sm, lc, ar, tid, NoHook{}, S::CS + (int)rank);
    __syncthreads();  // the transform's last exchange has been read
#pragma unroll
    for (int r = 0; r < C; ++r) sm[inv_out_elem<Cfg>(tid, r)] = x[0][r];
    cluster_sync();  // every part is in shared memory
    const uint32_t slice = rank * (NL / S::CS) + tid;
    uint64_t v[1][S::ITEMS][S::CS];
    split_inv_cross<S, 1, SP>(v, sm, 0, slice, lc, ar);
    unsigned long long *dst = reinterpret_cast<unsigned long long *>(sg.out + off + slice);
#pragma unroll
    for (int it = 0; it < S::ITEMS; ++it)
#pragma unroll
        for (int c = 0; c < S::CS; ++c) dst[it * T + c * NL] = v[0][it][c];
    cluster_sync();  // the peers have read this CTA's part
}

// output slots of a launch's products, by value
struct SlotList {
    uint32_t s[kSplitMaxProducts];
};

// one limb of a standalone product per cluster, a thread group per component:
//   out[slot][c] (+)= INTT(NTT(ct[j][c]) . pt[j])                              (App. C.1)
template <class S, bool SP>
__global__ void __cluster_dims__(S::CS, 1, 1) __launch_bounds__(S::THREADS, S::MINB)
k_product_split(const uint64_t *ct, const uint64_t *pt, uint64_t *out,
                const LimbConst *__restrict__ limbs, uint32_t L, int accumulate,
                const __grid_constant__ SlotList slots)
{
    static_assert(S::NG == 2 && S::NP == 1, "a group per component");
    using Cfg = typename S::Cfg;
    constexpr int C = S::C, T = S::T, NL = S::NL;
    constexpr size_t N = (size_t)1 << S::LOGN;
    extern __shared__ __align__(16) uint64_t sm[];  // [2][NL]
    const int tid = threadIdx.x % T;
    const uint32_t comp = threadIdx.x / T, rank = cluster_rank(), unit = blockIdx.x >> S::LOGP;
    const uint32_t j = unit / L, limb = unit - j * L;
    const LimbConst &lc = limbs[limb];
    const TwArith<SP> ar = tw_arith<SP>(lc);
    const int tmul = S::CS + (int)rank;
    const uint32_t slice = rank * (NL / S::CS) + tid;
    uint64_t *b = sm + comp * NL;
    cluster_sync();  // every CTA of the cluster is running before one writes into another
    pdl_begin();
    split_fwd_cross<S, 1, SP>(after_wait(ct) + ((size_t)(2 * j + comp) * L + limb) * N, 0, sm, comp * NL, slice, lc, ar);
    cluster_sync();  // this CTA's parts are complete
    uint64_t x[1][C];
#pragma unroll
    for (int r = 0; r < C; ++r) x[0][r] = b[tid + r * T];
    fwd_rounds<Cfg, 0, S::LOGP, SP>(x, b, lc.tw_f, nullptr, ar, tid, tmul);
    const ulonglong2 *w =
        reinterpret_cast<const ulonglong2 *>(after_wait(pt + ((size_t)j * L + limb) * N + rank * NL + tid * C));
#pragma unroll
    for (int r = 0; r < C; r += 2) {
        const ulonglong2 a = ld_data(w + r / 2);
        x[0][r] = mul_slot(ar, x[0][r], a.x, lc.r64, lc.r64_s);
        x[0][r + 1] = mul_slot(ar, x[0][r + 1], a.y, lc.r64, lc.r64_s);
    }
    inv_transform<Cfg, S::LOGP>(x, b, lc, ar, tid, NoHook{}, tmul);
    group_sync<Cfg>();  // the transform's last exchange has been read
#pragma unroll
    for (int r = 0; r < C; ++r) b[inv_out_elem<Cfg>(tid, r)] = x[0][r];
    cluster_sync();  // every part is in shared memory
    uint64_t v[1][S::ITEMS][S::CS];
    split_inv_cross<S, 1, SP>(v, sm, comp * NL, slice, lc, ar);
    uint64_t *dst = out + ((size_t)(2 * slots.s[j] + comp) * L + limb) * N + slice;
#pragma unroll
    for (int it = 0; it < S::ITEMS; ++it)
#pragma unroll
        for (int c = 0; c < S::CS; ++c) {
            uint64_t *d = dst + it * T + c * NL;
            *d = accumulate ? csub(*d + v[0][it][c], ar.q) : v[0][it][c];
        }
    cluster_sync();  // the peers have read this CTA's parts
}

}  // namespace hc
