// hc_keyswitch.cuh -- the key switch of a rotation as one kernel (hc_rotate.cu):
//   u[c][i] = INTT_i( sum_j NTT_i(d_j) . k_j[c][i] ),   c = 0, 1,
// d_j the limb-j digit of an already permuted c1, i one of the L+1 moduli of Q*p_sp.
//
// One cluster of 2^LOGP CTAs computes both components of one (ciphertext, modulus):
// the L digits are transformed where they stand, in the CTAs' shared memory, multiplied
// by the key and summed in registers, and the two sums are transformed back; digits and
// products never go to memory (L (L+1) + 2 (L+1) polynomials of a ciphertext written and
// read again by separate transform and multiply kernels).  A transform of N residues
// is split as in hc_split.cuh: the first LOGP forward stages pair residues N / 2^LOGP
// apart, each CTA computes them for its slice of the pairs and writes the results into
// the CTA that owns them (distributed shared memory), the rest is local to the CTA;
// the inverse runs the other way round.  2^LOGP CTAs per unit are for latency: the
// accumulator chain of one client has L+1 units a step.
// Bound by latency (few units: barriers of the cluster and the dependent products of one
// warp) or by the multiply pipe as the transforms are (many).  Measured on GB300, N = 8192,
// L = 3: a step of one ciphertext's chain 37 us as five kernels (digits, transform, product,
// transform, division), 15.6 us as this one and the division; a 3x3 Z_P layer of 32
// ciphertexts 1220 -> 1011 us.
//
// A digit is a residue below 2^50 and is taken as it stands: any representative modulo
// the unit's modulus gives the same canonical sum, and the transforms' bounds hold for
// inputs below 2^50 in both twiddle forms (folded: |.| <= (35 log2 N + 2) q < 2^59;
// Shoup: < 2^50 + 4 log2 N q < 2^56).  Sums of at most 7 products, folded: digits
// < 2^53, so V < 2^106, and reduce128_special's A2 < 2^28 still fits its word and leaves
// less than 3.25 * 2^50 < 4 q, which canon3 takes.
#pragma once

#include <atomic>

#include "hc_split.cuh"

namespace hc {

// the other stages of NP digits in the buffers b, b + NL; a thread's residues (elements
// tid*C + r) end up in its own swizzled positions
template <class S, int NP, bool SP>
__device__ __forceinline__ void ks_fwd_local(uint64_t *b, const LimbConst &lc, const TwArith<SP> &ar, int tid,
                                             int tmul)
{
    using Cfg = typename S::template CfgP<NP>;
    constexpr int C = Cfg::C, T = Cfg::T, NL = Cfg::N;
    uint64_t x[NP][C];
#pragma unroll
    for (int r = 0; r < C; ++r)
#pragma unroll
        for (int p = 0; p < NP; ++p) x[p][r] = b[p * NL + tid + r * T];
    fwd_rounds<Cfg, 0, S::LOGP, SP>(x, b, lc.tw_f, nullptr, ar, tid, tmul);
    // the last exchange has been read: by the warp's own threads when it was warp-local
    xsync<Cfg, fwd_round_local<Cfg, Cfg::NROUNDS - 2>()>();
#pragma unroll
    for (int r = 0; r < C; ++r)
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if constexpr (SP)  // [0, 2^53), as the sums want it
                b[p * NL + spos_at<Cfg>(tid * C, r)] = ar.fold(x[p][r] + 2048 * ar.q);
            else
                b[p * NL + spos_at<Cfg>(tid * C, r)] = x[p][r];
        }
}

// a buffer per digit, or per component
template <class S>
size_t ks_smem(uint32_t L)
{
    return (size_t)(L < 2 ? 2 : L) * S::NL * sizeof(uint64_t);
}

template <class S, bool SP>
__global__ void __cluster_dims__(S::CS, 1, 1) __launch_bounds__(S::THREADS, S::MINB)
k_ks_switch(const KsArgs args)
{
    using Cfg = typename S::template CfgP<S::NP>;
    constexpr int LOGP = S::LOGP, CS = S::CS, C = S::C, T = S::T, NL = S::NL, ITEMS = S::ITEMS, NG = S::NG, NP = S::NP;
    constexpr size_t N = (size_t)1 << S::LOGN;
    static_assert(S::NG * S::NP >= 2, "both components at once");
    extern __shared__ __align__(16) uint64_t sm[];  // [max(L, 2)][NL]
    const int tid = threadIdx.x % T;
    const uint32_t first = threadIdx.x / T * NP;  // the group's first digit and component
    const uint32_t rank = cluster_rank(), unit = blockIdx.x >> LOGP;
    const uint32_t L = args.L, L1 = L + 1, ct = unit / L1, i = unit - ct * L1;
    const LimbConst &lc = args.lqp[i];
    const TwArith<SP> ar = tw_arith<SP>(lc);
    const int tmul = CS + (int)rank;
    const uint32_t slice = rank * (NL / CS) + tid;  // this thread's first pair of the cross stages
    cluster_sync();  // every CTA of the cluster is running before one writes into another
    pdl_begin();

    const uint64_t *c1 = after_wait(args.a) + (size_t)(2 * ct + 1) * L * N;
    for (uint32_t j = first; j < L; j += NG * NP) {
        if (j + NP <= L)
            split_fwd_cross<S, NP, SP>(c1 + j * N, N, sm, j * NL, slice, lc, ar);
        else
            split_fwd_cross<S, 1, SP>(c1 + j * N, N, sm, j * NL, slice, lc, ar);
    }
    cluster_sync();  // this CTA's parts of the digits are complete
    for (uint32_t j = first; j < L; j += NG * NP) {
        if (j + NP <= L)
            ks_fwd_local<S, NP, SP>(sm + j * NL, lc, ar, tid, tmul);
        else
            ks_fwd_local<S, 1, SP>(sm + j * NL, lc, ar, tid, tmul);
    }
    if constexpr (NG > 1) __syncthreads();  // every group's digits are there

    // sums over the digits of components first .. first + NP - 1
    uint64_t x[NP][C];
    if (first < 2) {
        constexpr int E = 4 / NP;  // residues at a time
        const uint64_t *key = args.key + ((size_t)first * L1 + i) * N + rank * NL + tid * C;
#pragma unroll
        for (int h = 0; h < C; h += E) {
            MacAcc acc[NP][E];
#pragma unroll
            for (int p = 0; p < NP; ++p)
#pragma unroll
                for (int e = 0; e < E; ++e) mac_zero(acc[p][e]);
            for (uint32_t j = 0; j < L; ++j) {
                const uint64_t *b = sm + j * NL;
#pragma unroll
                for (int p = 0; p < NP; ++p)
#pragma unroll
                    for (int e = 0; e < E; e += 2) {
                        const ulonglong2 k = __ldg(
                            reinterpret_cast<const ulonglong2 *>(key + (size_t)(2 * j + p) * L1 * N + h + e));
                        mac_add(acc[p][e], b[spos_at<Cfg>(tid * C, h + e)], k.x);
                        mac_add(acc[p][e + 1], b[spos_at<Cfg>(tid * C, h + e + 1)], k.y);
                    }
            }
#pragma unroll
            for (int p = 0; p < NP; ++p)
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    if constexpr (SP)
                        x[p][h + e] = mac_reduce_special(acc[p][e], ar.q, ar.c);
                    else
                        x[p][h + e] = mac_reduce(acc[p][e], ar.q, ar.nq, lc.r64, lc.r64_s, ar.ones);
                }
        }
    }
    if constexpr (NG > 1) __syncthreads();  // both components have read every digit
    // inverse: the CTA's part, then the last LOGP stages across the cluster
    if (first < 2) {
        uint64_t *b = sm + first * NL;
        inv_transform<Cfg, LOGP>(x, b, lc, ar, tid, NoHook{}, tmul);
        group_sync<Cfg>();  // the transform's last exchange has been read
#pragma unroll
        for (int r = 0; r < C; ++r)
#pragma unroll
            for (int p = 0; p < NP; ++p) b[p * NL + inv_out_elem<Cfg>(tid, r)] = x[p][r];
    }
    cluster_sync();  // every part is in shared memory
    if (first < 2) {
        uint64_t v[NP][ITEMS][CS];
        split_inv_cross<S, NP, SP>(v, sm, first * NL, slice, lc, ar);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            uint64_t *u = args.u + ((size_t)(2 * ct + first + p) * L1 + i) * N + slice;
#pragma unroll
            for (int it = 0; it < ITEMS; ++it)
#pragma unroll
                for (int c = 0; c < CS; ++c) u[it * T + c * NL] = v[p][it][c];
        }
    }
    cluster_sync();  // the peers have read this CTA's parts
}

// one launch; dynamic shared memory grows with the limb count
template <class S, bool SP>
hc_status run_ks_switch(const KsArgs &a, size_t n, cudaStream_t s)
{
    auto kern = k_ks_switch<S, SP>;
    static std::atomic<uint32_t> done{0};
    int dev = 0;
    cudaGetDevice(&dev);
    const uint32_t bit = 1u << (dev & 31);
    if (!(done.load(std::memory_order_relaxed) & bit)) {
        const cudaError_t e =
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ks_smem<S>(kMaxLimbs - 1));
        if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(k_ks_switch)");
        done.fetch_or(bit);
    }
    const size_t ctas = n * (a.L + 1) * S::CS;
    if (ctas > 0x7fffffffu) return set_error(HC_ERR_INVALID_ARG, "batch too large");
    ProfileScope ps("k_ks_switch", s);
    const cudaError_t e = launch_programmatic(kern, dim3((unsigned)ctas), dim3(S::THREADS), ks_smem<S>(a.L), s, true, a);
    return e == cudaSuccess ? HC_OK : cuda_error(e, "launch k_ks_switch");
}

// Up to two latency CTAs per SM, a thread group per digit (two groups at N = 16384, where a
// thread has no registers for more); beyond, 2048 residues a CTA.  Measured on GB300, a
// whole step (key switch and division) of n ciphertexts, latency / throughput shape, us:
//   N = 8192, L = 3:   n = 1: 15.6 / 26.8   n = 8: 46.8 / 52.9   n = 16: 81.1 / 59.6
//   N = 4096, L = 2:   n = 1: 10.8 / 17.7   n = 8: 21.8 / 39.0   n = 16: 39.8 / 40.9
//   N = 16384, L = 4:  n = 1: 26.1 / 53.0   n = 6: 65.5 / 70.8   n = 8: 93.1 / 76.2
template <int LOGN, bool SP>
hc_status launch_ks_n(const KsArgs &a, size_t n, uint32_t sms, cudaStream_t s)
{
    const bool few = 8 * n * (a.L + 1) <= 2 * (size_t)sms;
    if constexpr (LOGN < 14) {
        if (few) return run_ks_switch<SplitShape<LOGN, 3, 4, 1, 3, 8>, SP>(a, n, s);
    } else {
        if (few) return run_ks_switch<SplitShape<LOGN, 3, 2, 1, 3, 16>, SP>(a, n, s);
    }
    return run_ks_switch<SplitShape<LOGN, LOGN - 11, 1, 2>, SP>(a, n, s);
}

}  // namespace hc
