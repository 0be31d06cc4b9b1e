// hc_ntt.cuh -- register-resident negacyclic NTT engine for one CTA.
//
// A CTA transforms NP polynomials of N = 2^LOGN residues (NP = 2: both
// components of one ciphertext limb, sharing every twiddle load) with
// T = N / C threads; each thread holds C = 2^LOGC residues of every
// polynomial in registers.  The log2 N butterfly stages run in rounds of
// LOGC stages entirely inside registers; between rounds the CTA exchanges
// data through shared memory (one write, one read per element).
//
// Forward (App. C.1, natural order in, slot order out): Cooley-Tukey stages
// with the psi powers merged into the twiddles (Longa & Naehrig 2016); stage
// s has 2^s groups of 2t = N / 2^s elements, group i uses psi^rev(2^s + i).
// Inverse: Gentleman-Sande stages, stage s (half distance 2^s) has
// N / 2^(s+1) groups, group i uses psi^-rev(N/2^(s+1) + i); N^-1 is merged
// into the last stage.
//
// Twiddle products (TwArith): limbs with q = 2^50 - c, c < 2^22 (SP), multiply by
// folding, on signed lazy values; the others by Shoup's method, on unsigned ones.  A
// context whose limbs are all of that kind holds its tables in the folded form (16
// bytes per twiddle either way) and its launches take the SP kernels.  Both forms in one
// kernel, chosen per CTA, cost the folded one registers: 112.8 instead of 97.7 us for
// 1536 inverse transforms at N = 8192.
// Lazy bounds (q < 2^50, N <= 2^14; products < 4q by Shoup, |.| <= 35 q folded):
//   forward: inputs < q; each stage adds a product -> outputs < (4 log2 N + 1) q < 2^56
//            by Shoup, |.| <= (35 log2 N + 1) q < 2^59 folded
//   inverse, Shoup: inputs < q; stage 0 corrects its products to < 2q, so stage-s
//            inputs are < 2^s q and X - Y + 2^s q < 2^(s+1) q <= 2^64; the last
//            stage's Shoup steps (N^-1 merged) and two corrections give
//            canonical output.
//   inverse, folded: sums double and products restart at 35 q, so within a round only
//            the registers that were sums throughout, or were products in the first
//            stages, grow large; those above what the next round may take
//            (inv_fold_limit) are folded below 5 q: at most four of a round's 32.
// Twiddle loads: in the inverse's first round and the forward's last round
// every thread needs its own twiddles (N/2 distinct ones in the inverse's
// first stage); read from the natural tables a warp's 32 loads would hit 32
// lines, so those rounds read context tables rearranged so that a warp's
// loads are consecutive (LimbConst::tw_r); the other rounds share each
// twiddle among neighbouring threads and read the natural tables.
// Shared-memory layout: element e of polynomial p lives at word p * SW + spos(e),
// e ^ ((e >> LOGC) & 15) below N = 16384, e + (e >> LOGC) there (one word of padding after
// every C).  Either makes every 8-byte access pattern below conflict-free (the 16 threads
// of each half-warp touch 16 distinct bank pairs).  The padded position of a thread's first
// element plus a constant is the position of the others (spos_at), so that an access is one
// instruction with an immediate offset, where the XOR takes two more.  Measured on GB300,
// XOR / padded, us: N = 16384, 2048 limbs forward 295 / 288, inverse 275 / 272, 800 products
// 1785 / 1707; N = 8192, 1536 limbs inverse 93 / 95; N = 4096, 4096 limbs inverse 99 / 102;
// forward about even: hence the line.  Eight residues per thread would conflict padded.
#pragma once

#include <type_traits>

#include "hc_arith.cuh"
#include "hc_internal.h"

namespace hc {

template <int LOGN_, int LOGC_, int NP_, int MINB_ = 1, int GROUPS_ = 1>
struct NttCfg {
    static constexpr int LOGN = LOGN_;
    static constexpr int LOGC = LOGC_;
    static constexpr int NP = NP_;
    static constexpr int MINB = MINB_;  // CTAs per SM the register budget is sized for
    static constexpr int GROUPS = GROUPS_;  // groups of T threads that run transforms of their own side by side
    static constexpr int N = 1 << LOGN;
    static constexpr int C = 1 << LOGC;
    static constexpr int T = N / C;
    static constexpr int NROUNDS = (LOGN + LOGC - 1) / LOGC;
    static constexpr bool PADDED = LOGN >= 14 && LOGC >= 4;
    static constexpr int SW = PADDED ? N + (N >> LOGC) : N;  // shared words per polynomial
    static constexpr size_t SMEM_BYTES = (size_t)NP * SW * sizeof(uint64_t);
    static_assert(LOGC >= 2 && LOGC <= LOGN, "bad radix");
};

template <class Cfg>
__host__ __device__ __forceinline__ constexpr int spos(int e)
{
    return Cfg::PADDED ? e + (e >> Cfg::LOGC) : e ^ ((e >> Cfg::LOGC) & 15);
}
// position of element base + off: base the thread's first element of an access pattern, off
// a constant, base mod C + off mod C < C
template <class Cfg>
__device__ __forceinline__ int spos_at(int base, int off)
{
    return Cfg::PADDED ? spos<Cfg>(base) + spos<Cfg>(off) : spos<Cfg>(base + off);
}

template <class Cfg, int R>
struct RoundShape {
    static constexpr int S0 = R * Cfg::LOGC;
    static constexpr int K = (Cfg::LOGN - S0) < Cfg::LOGC ? (Cfg::LOGN - S0) : Cfg::LOGC;
    static constexpr int KK = 1 << K;
    static constexpr int SUBS = Cfg::C >> K;  // sub-transforms per thread
};

// ---- element owned by (thread, register slot r = v*KK + j) in each round ------------
// As base (of the thread) plus offset (constant after unrolling), for spos_at.
// forward round: sub-transform u = tid*SUBS + v covers, at stride S = N >> (S0+K),
// the KK elements (u / S) * (N >> S0) + (u % S) + j*S.
template <class Cfg, int R>
__device__ __forceinline__ int fwd_base(int tid)
{
    using RS = RoundShape<Cfg, R>;
    constexpr int S = Cfg::N >> (RS::S0 + RS::K);
    static_assert(RS::SUBS == 1 || S == 1, "only the last round has several sub-transforms");
    return S == 1 ? tid * Cfg::C : (tid / S) * (Cfg::N >> RS::S0) + tid % S;
}
template <class Cfg, int R>
__device__ __forceinline__ int fwd_off(int r)
{
    using RS = RoundShape<Cfg, R>;
    constexpr int S = Cfg::N >> (RS::S0 + RS::K);
    return S == 1 ? r : r * S;
}
// inverse round: sub-transform u = tid + v*T covers, at stride S = 2^S0, the KK
// elements (u / S) * (S << K) + (u % S) + j*S.
template <class Cfg, int R>
__device__ __forceinline__ int inv_base(int tid)
{
    using RS = RoundShape<Cfg, R>;
    constexpr int S = 1 << RS::S0;
    return (tid / S) * (S << RS::K) + tid % S;
}
template <class Cfg, int R>
__device__ __forceinline__ int inv_off(int r)
{
    using RS = RoundShape<Cfg, R>;
    constexpr int S = 1 << RS::S0;
    static_assert(Cfg::T % S == 0 || S == Cfg::N >> RS::K, "a sub-transform's blocks are whole");
    const int v = r >> RS::K, j = r & (RS::KK - 1);
    return (Cfg::T % S == 0 ? v * (Cfg::T << RS::K) : v * Cfg::T) + j * S;
}

// ---- compile-time loop -------------------------------------------------------------
template <int I, int END, class F>
__device__ __forceinline__ void static_for(F &&f)
{
    if constexpr (I < END) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, END>(f);
    }
}

// ---- one forward round: K Cooley-Tukey stages in registers ---------------------
// PART > 0: the transform is one of the 2^PART parts of a larger transform after that
// transform's first PART stages (see k_ntt_fwd_pair, hc_split.cuh): local stage s,
// group i uses the full table's entry tmul*2^s + i, tmul = 2^PART + the part's
// index; every round reads the natural table.
template <class Cfg, int R, int SIG, int PART, bool SP>
__device__ __forceinline__ void fwd_stage(uint64_t (&x)[Cfg::NP][Cfg::C], const ulonglong2 *__restrict__ tw,
                                          const ulonglong2 *__restrict__ twr, const TwArith<SP> &ar, int v, int g0,
                                          int tid, int tmul)
{
    using RS = RoundShape<Cfg, R>;
    static_assert(Cfg::LOGC >= 3 && Cfg::LOGC <= 5, "last-round tables exist for LOGC = 3, 4, 5");
    constexpr int half = RS::KK >> (SIG + 1);
    constexpr bool last = R == Cfg::NROUNDS - 1 && PART == 0;  // every thread has its own twiddles (g0 = tid*SUBS + v)
#pragma unroll
    for (int lam = 0; lam < (1 << SIG); ++lam) {
        // last round: the rearranged table, stage S0 + SIG at [2^(S0+SIG) - 2^S0],
        // entry ((v << SIG) + lam)*T + tid, so that a warp reads consecutive entries
        const ulonglong2 w =
            last ? __ldg(twr + (size_t)(3 + Cfg::LOGC - 3) * Cfg::N + ((1 << (RS::S0 + SIG)) - (1 << RS::S0)) +
                         ((v << SIG) + lam) * Cfg::T + tid)
                 : __ldg(tw + ((PART ? tmul : 1) << (RS::S0 + SIG)) + (g0 << SIG) + lam);
#pragma unroll
        for (int jj = 0; jj < half; ++jj) {
            const int j = v * RS::KK + lam * 2 * half + jj;
#pragma unroll
            for (int p = 0; p < Cfg::NP; ++p) {
                const uint64_t X = x[p][j];
                const uint64_t t = ar.mul(x[p][j + half], w);
                x[p][j] = X + t;
                x[p][j + half] = ar.sub(X, t);
            }
        }
    }
}

template <class Cfg, int R, int PART, bool SP>
__device__ __forceinline__ void fwd_round(uint64_t (&x)[Cfg::NP][Cfg::C], const ulonglong2 *__restrict__ tw,
                                          const ulonglong2 *__restrict__ twr, const TwArith<SP> &ar, int tid, int tmul)
{
    using RS = RoundShape<Cfg, R>;
    constexpr int S = Cfg::N >> (RS::S0 + RS::K);
    static_for<0, RS::SUBS>([&](auto vc) {
        constexpr int v = decltype(vc)::value;
        const int g0 = (tid * RS::SUBS + v) / S;
        static_for<0, RS::K>([&](auto sc) {
            fwd_stage<Cfg, R, decltype(sc)::value, PART, SP>(x, tw, twr, ar, v, g0, tid, tmul);
        });
    });
}

// ---- one inverse round: K Gentleman-Sande stages in registers ------------------
// PART > 0: the transform is one of the 2^PART parts of a larger transform, before
// that transform's last PART stages (see hc_split.cuh): stage s, group
// i uses the full table's entry tmul*(N >> (s+1)) + i (N this transform's size, tmul =
// 2^PART + the part's index); every round reads the natural table and no stage is the
// last.
// Bounds, in multiples of q, of the folded form (values in the Shoup form follow 2^s).
// Between rounds a register may hold at most inv_fold_limit: the next round's K stages
// double it K - 1 times before the last X - Y, which must stay below 2^63 in magnitude,
// and 2 * 4096 q < 2^63.
template <class Cfg, int R, int PART>
constexpr uint64_t inv_fold_limit()
{
    if constexpr (R + 1 < Cfg::NROUNDS)
        return 4096u >> (RoundShape<Cfg, R + 1>::K - 1);
    else
        return 4096u >> (PART > 0 ? PART - 1 : 0);  // PART more stages, by the caller
}
// register j (of a sub-transform) after a round of K stages on inputs <= b q: j = 0 was a
// sum in every stage; else j's top bit is the stage of its last product
constexpr uint64_t inv_reg_bound(uint64_t b, int K, int j)
{
    if (j == 0) return b << K;
    int h = 0;
    while ((j >> h) > 1) ++h;
    return kFoldMax << (K - 1 - h);
}
template <class Cfg, int R, int PART>
constexpr uint64_t inv_in_bound()  // inputs of round R
{
    if constexpr (R == 0) {
        return 1;
    } else {
        uint64_t m = 0;
        for (int j = 0; j < RoundShape<Cfg, R - 1>::KK; ++j) {
            uint64_t b = inv_reg_bound(inv_in_bound<Cfg, R - 1, PART>(), RoundShape<Cfg, R - 1>::K, j);
            if (b > inv_fold_limit<Cfg, R - 1, PART>()) b = 5;
            if (b > m) m = b;
        }
        return m;
    }
}
// bound of the inputs of stage SIG of round R
template <class Cfg, int R, int SIG, int PART, bool SP>
constexpr uint64_t inv_stage_bound()
{
    if constexpr (!SP) {
        return 1ull << (RoundShape<Cfg, R>::S0 + SIG);
    } else {
        const uint64_t b = inv_in_bound<Cfg, R, PART>() << SIG;
        const uint64_t p = SIG > 0 ? kFoldMax << (SIG - 1) : 0;
        return b > p ? b : p;
    }
}

template <class Cfg, int R, int SIG, int PART, bool SP>
__device__ __forceinline__ void inv_stage(uint64_t (&x)[Cfg::NP][Cfg::C], const LimbConst &lc, const TwArith<SP> &ar,
                                          const ulonglong2 *__restrict__ tw, int v, int blk, int tmul)
{
    using RS = RoundShape<Cfg, R>;
    static_assert(Cfg::LOGC >= 3 && Cfg::LOGC <= 5, "first-round tables exist for LOGC = 3, 4, 5");
    constexpr int s = RS::S0 + SIG;  // global stage
    constexpr int dist = 1 << SIG;
    constexpr int ngrp = RS::KK >> (SIG + 1);
    constexpr uint64_t bound = inv_stage_bound<Cfg, R, SIG, PART, SP>();
    static_assert(bound <= (SP ? kFoldStage : 8192), "differences must fit 64 bits, and div_canon's shift");
    const uint64_t q = ar.q;
    const uint64_t qs = q * bound;    // bound of the stage's inputs
    if constexpr (s == Cfg::LOGN - 1 && PART == 0) {
        // last stage: N^-1 merged into both outputs, canonical result
        const ulonglong2 wn = make_ulonglong2(lc.ninv, lc.ninv_s), wnw = make_ulonglong2(lc.ninvw, lc.ninvw_s);
#pragma unroll
        for (int grp = 0; grp < ngrp; ++grp) {
#pragma unroll
            for (int jj = 0; jj < dist; ++jj) {
                const int j = v * RS::KK + grp * 2 * dist + jj;
#pragma unroll
                for (int p = 0; p < Cfg::NP; ++p) {
                    const uint64_t X = x[p][j], Y = x[p][j + dist];
                    x[p][j] = ar.template div_canon<Cfg::LOGN>(X + Y, wn);
                    x[p][j + dist] = ar.mul_canon(ar.sub(X, Y, qs), wnw);
                }
            }
        }
    } else {
#pragma unroll
        for (int grp = 0; grp < ngrp; ++grp) {
            // first round: blk is the thread index, and the rearranged table gives the
            // warp consecutive entries; later rounds share each twiddle across threads
            const ulonglong2 w =
                R == 0 && PART == 0
                    ? __ldg(lc.tw_r + (size_t)(Cfg::LOGC - 3) * Cfg::N + (Cfg::N - (Cfg::N >> s)) + grp * Cfg::T + blk)
                    : __ldg(tw + (PART ? tmul : 1) * (Cfg::N >> (s + 1)) + blk * ngrp + grp);
#pragma unroll
            for (int jj = 0; jj < dist; ++jj) {
                const int j = v * RS::KK + grp * 2 * dist + jj;
#pragma unroll
                for (int p = 0; p < Cfg::NP; ++p) {
                    const uint64_t X = x[p][j], Y = x[p][j + dist];
                    x[p][j] = X + Y;
                    const uint64_t t = ar.mul(ar.sub(X, Y, qs), w);
                    x[p][j + dist] = !SP && s == 0 ? csub(t, 2 * q) : t;
                }
            }
        }
    }
}

template <class Cfg, int R, int PART, bool SP>
__device__ __forceinline__ void inv_round(uint64_t (&x)[Cfg::NP][Cfg::C], const LimbConst &lc, const TwArith<SP> &ar,
                                          const ulonglong2 *__restrict__ tw, int tid, int tmul)
{
    using RS = RoundShape<Cfg, R>;
    constexpr int S = 1 << RS::S0;
    static_for<0, RS::SUBS>([&](auto vc) {
        constexpr int v = decltype(vc)::value;
        const int blk = (tid + v * Cfg::T) / S;
        static_for<0, RS::K>([&](auto sc) {
            inv_stage<Cfg, R, decltype(sc)::value, PART, SP>(x, lc, ar, tw, v, blk, tmul);
        });
        if constexpr (SP && (R + 1 < Cfg::NROUNDS || PART > 0))
            static_for<0, RS::KK>([&](auto jc) {
                constexpr int j = decltype(jc)::value;
                if constexpr (inv_reg_bound(inv_in_bound<Cfg, R, PART>(), RS::K, j) > inv_fold_limit<Cfg, R, PART>())
#pragma unroll
                    for (int p = 0; p < Cfg::NP; ++p) x[p][v * RS::KK + j] = ar.fold(x[p][v * RS::KK + j]);
            });
    });
}

// ---- warp-local rounds ---------------------------------------------------------------
// A round is warp-local when every thread's elements in it lie in its own warp's
// block of 32*C consecutive elements (warp w: [32wC, 32(w+1)C)).  An exchange
// between two warp-local rounds moves data only within each warp's block, so a
// warp barrier replaces the CTA barrier on both of its sides: the writes go to
// the warp's own block, whose last readers (the previous round's layout) were
// the warp's own threads.  Inverse round R (u = tid when it has one
// sub-transform per thread, stride S = C^R): local iff it has one sub-transform
// per thread and C^R <= 32 -- rounds 0 and 1 for every shape here.  Forward
// round R (stride N >> (RC + K) over blocks of N >> RC): local iff
// log2 N - R log2 C <= 5 + log2 C -- the last two rounds (three for some
// shapes).  Checked for every shape on a CPU model of these layouts.
#ifndef HC_WARP_LOCAL_XCHG
#define HC_WARP_LOCAL_XCHG 1
#endif
template <class Cfg, int R>
constexpr bool inv_round_local()
{
    return RoundShape<Cfg, R>::K == Cfg::LOGC && R * Cfg::LOGC <= 5;
}
template <class Cfg, int R>
constexpr bool fwd_round_local()
{
    return Cfg::LOGN - R * Cfg::LOGC <= 5 + Cfg::LOGC;
}
// the threads of one transform: the CTA, or one of its groups (named barriers 1 ...)
template <class Cfg>
__device__ __forceinline__ void group_sync()
{
    if constexpr (Cfg::GROUPS == 1)
        __syncthreads();
    else  // barrier numbers as constants: a register would reserve all sixteen
        static_for<0, Cfg::GROUPS>([](auto gc) {
            constexpr int g = decltype(gc)::value;
            if (threadIdx.x / Cfg::T == g) asm volatile("bar.sync %0, %1;" ::"n"(1 + g), "n"(Cfg::T) : "memory");
        });
}
template <class Cfg, bool WARP>
__device__ __forceinline__ void xsync()
{
    if constexpr (WARP && HC_WARP_LOCAL_XCHG)
        __syncwarp();
    else
        group_sync<Cfg>();
}

// ---- exchanges through shared memory ---------------------------------------------
template <class Cfg, int RFROM>
__device__ __forceinline__ void fwd_exchange(uint64_t (&x)[Cfg::NP][Cfg::C], uint64_t *sm, int tid)
{
    constexpr bool local = fwd_round_local<Cfg, RFROM>() && fwd_round_local<Cfg, RFROM + 1>();
    xsync<Cfg, local>();
#pragma unroll
    for (int r = 0; r < Cfg::C; ++r) {
        const int e = spos_at<Cfg>(fwd_base<Cfg, RFROM>(tid), fwd_off<Cfg, RFROM>(r));
#pragma unroll
        for (int p = 0; p < Cfg::NP; ++p) sm[p * Cfg::SW + e] = x[p][r];
    }
    xsync<Cfg, local>();
#pragma unroll
    for (int r = 0; r < Cfg::C; ++r) {
        const int e = spos_at<Cfg>(fwd_base<Cfg, RFROM + 1>(tid), fwd_off<Cfg, RFROM + 1>(r));
#pragma unroll
        for (int p = 0; p < Cfg::NP; ++p) x[p][r] = sm[p * Cfg::SW + e];
    }
}

template <class Cfg, int RFROM>
__device__ __forceinline__ void inv_exchange(uint64_t (&x)[Cfg::NP][Cfg::C], uint64_t *sm, int tid)
{
    constexpr bool local = inv_round_local<Cfg, RFROM>() && inv_round_local<Cfg, RFROM + 1>();
    xsync<Cfg, local>();
#pragma unroll
    for (int r = 0; r < Cfg::C; ++r) {
        const int e = spos_at<Cfg>(inv_base<Cfg, RFROM>(tid), inv_off<Cfg, RFROM>(r));
#pragma unroll
        for (int p = 0; p < Cfg::NP; ++p) sm[p * Cfg::SW + e] = x[p][r];
    }
    xsync<Cfg, local>();
#pragma unroll
    for (int r = 0; r < Cfg::C; ++r) {
        const int e = spos_at<Cfg>(inv_base<Cfg, RFROM + 1>(tid), inv_off<Cfg, RFROM + 1>(r));
#pragma unroll
        for (int p = 0; p < Cfg::NP; ++p) x[p][r] = sm[p * Cfg::SW + e];
    }
}

// ---- whole transforms -----------------------------------------------------------
// forward: x holds the round-0 layout (element tid + r*T) on entry and the
// last-round layout (element tid*C + r, contiguous) on exit.
template <class Cfg, int R, int PART, bool SP>
__device__ __forceinline__ void fwd_rounds(uint64_t (&x)[Cfg::NP][Cfg::C], uint64_t *sm,
                                           const ulonglong2 *__restrict__ tw, const ulonglong2 *__restrict__ twr,
                                           const TwArith<SP> &ar, int tid, int tmul)
{
    fwd_round<Cfg, R, PART, SP>(x, tw, twr, ar, tid, tmul);
    if constexpr (R + 1 < Cfg::NROUNDS) {
        fwd_exchange<Cfg, R>(x, sm, tid);
        fwd_rounds<Cfg, R + 1, PART, SP>(x, sm, tw, twr, ar, tid, tmul);
    }
}

template <class Cfg, bool SP>
__device__ __forceinline__ void fwd_transform(uint64_t (&x)[Cfg::NP][Cfg::C], uint64_t *sm, const LimbConst &lc,
                                              const TwArith<SP> &ar, int tid)
{
    fwd_rounds<Cfg, 0, false, SP>(x, sm, lc.tw_f, lc.tw_r, ar, tid, 1);
}

struct NoHook {
    __device__ __forceinline__ void operator()() const {}
};

// inverse: x holds element tid*C + r (contiguous) on entry, canonical values
// < q; on exit the last-round layout (element tid + r'*T for the slot order of
// inv_base, inv_off), canonical.  The first exchange synchronises the warp only: since
// the caller's last CTA barrier, no thread may have accessed shared memory
// outside its own warp's block of 32*C elements (every caller's last accesses
// are its reads of the round-0 layout, element tid*C + r).  hook() runs (in every thread) right before the last
// round, once this transform has finished with shared memory: after its last
// exchange, or after the caller's reads when there is one round only.
template <class Cfg, int R, class Hook, int PART, bool SP>
__device__ __forceinline__ void inv_rounds(uint64_t (&x)[Cfg::NP][Cfg::C], uint64_t *sm, const LimbConst &lc,
                                           const TwArith<SP> &ar, int tid, const Hook &hook, int tmul)
{
    if constexpr (R + 1 == Cfg::NROUNDS) hook();
    inv_round<Cfg, R, PART, SP>(x, lc, ar, lc.tw_i, tid, tmul);
    if constexpr (R + 1 < Cfg::NROUNDS) {
        inv_exchange<Cfg, R>(x, sm, tid);
        inv_rounds<Cfg, R + 1, Hook, PART, SP>(x, sm, lc, ar, tid, hook, tmul);
    }
}

template <class Cfg, int PART = 0, bool SP, class Hook = NoHook>
__device__ __forceinline__ void inv_transform(uint64_t (&x)[Cfg::NP][Cfg::C], uint64_t *sm, const LimbConst &lc,
                                              const TwArith<SP> &ar, int tid, const Hook &hook = Hook{}, int tmul = 1)
{
    inv_rounds<Cfg, 0, Hook, PART, SP>(x, sm, lc, ar, tid, hook, tmul);
}

// the last inverse-round layout: slot r = v*KK + j holds element
// tid + T*(v + j*SUBS)  (coalesced across the warp)
template <class Cfg>
__device__ __forceinline__ int inv_out_elem(int tid, int r)
{
    using RS = RoundShape<Cfg, Cfg::NROUNDS - 1>;
    const int v = r >> RS::K, j = r & (RS::KK - 1);
    return tid + Cfg::T * (v + j * RS::SUBS);
}

// the limb's arithmetic (SP as its context's tables, hc_ctx::fold)
template <bool SP>
__device__ __forceinline__ TwArith<SP> tw_arith(const LimbConst &lc)
{
    return TwArith<SP>(lc.q, lc.special_c, lc.one_s);
}

}  // namespace hc
