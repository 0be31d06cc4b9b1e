// hc_mac.cuh -- the blocked NTT-domain convolution MAC (Sec. 6.2) as one CTA
// task, shared by the stand-alone MAC kernel and the fused persistent
// convolution kernel:
//   Y[m*B+b][c] = sum_g W[m*G+g] . X[g*B+b][c]      (slot-wise, mod q_limb)
//
// A task owns one chunk of KC slots of one limb for every input ciphertext
// and the output channels [m0, m1).  The input chunk (G*2B rows of KC slots)
// is fetched once into shared memory by TMA bulk copies; the weight slices
// stream through a ring of kMacStages shared-memory stages of MS channels
// each (MS*G rows of KC slots), refilled while the other stages are in use.
// Each weight slot is therefore read from memory once and each input slot
// once per channel group.  Thread (k, h) owns slot k0 + k; the NT / KC row groups h take
// the tasks' (channel pair, block) tiles in turn: two channels by the two components of
// one spatial block, so that two input and two weight slots read from shared memory feed
// four products.  The input chunk is cut at 2^25 in place once it has arrived (hc_arith.cuh,
// MacAcc25), a weight slot when it is read.
// Bound by the issue slots and the multiply pipe (12 cycles of that pipe a product plus 24
// a reduction).  Measured on GB300, 56x56x64 layer (G = 8, B = 4): 130 -> 107 us with the
// cut at 2^25 and stages of two channels.
//
// A stage is handed back warp by warp (an "empty" mbarrier of one arrival per warp) and
// refilled by thread 0, so that warps run up to kMacStages apart without a CTA barrier.
// The ring's mbarriers live for the whole CTA; a MacRing carries their
// phase counters from one task to the next.  Waits are bounded: a wait that
// runs out sets err = 2, drains the task's copies in flight (bounded) and
// makes the task return false.
#pragma once

#include <type_traits>

#include "hc_arith.cuh"
#include "hc_async.cuh"
#include "hc_internal.h"

namespace hc {

constexpr int kMacStages = 3;
constexpr int kMacKC = 64;

// mbarriers of a CTA: the input chunk, then per stage "full" and "empty"
constexpr int kMacBars = 1 + 2 * kMacStages;

struct MacRing {
    uint32_t gi;    // weight stages loaded and consumed so far by this CTA
    uint32_t xuse;  // input chunks loaded so far by this CTA
};

// by one thread, before a CTA barrier
template <int NT>
__device__ __forceinline__ void mac_bars_init(uint64_t *bars)
{
    for (int i = 0; i < 1 + kMacStages; ++i) mbar_init(&bars[i], 1);
    for (int i = 0; i < kMacStages; ++i) mbar_init(&bars[1 + kMacStages + i], NT / 32);
    mbar_fence_init();
}

// The caller has synchronised the CTA since its last generic shared-memory access.
template <int KC, int NT>
__device__ __forceinline__ bool mac_task(const MacSeg &sg, uint32_t chunk, uint32_t limb, uint32_t m0, uint32_t m1,
                                         uint64_t *dsm, uint64_t *bars, MacRing &ring, int *err)
{
    constexpr int H = NT / KC;
    constexpr uint32_t ROW_BYTES = KC * sizeof(uint64_t);
    static_assert(NT % KC == 0 && KC % 32 == 0, "whole warps per row group");
    const uint32_t N = sg.N, L = sg.L, G = sg.G, B = sg.B, MS = sg.MS;
    const uint32_t P = 2 * B, rows = G * P, SR = MS * G;
    uint64_t *xs = dsm;                          // [rows][KC]
    uint64_t *ws = dsm + (size_t)rows * KC;      // [kMacStages][SR][KC]
    const uint32_t k0 = chunk * KC;
    const uint32_t nm = m1 > m0 ? m1 - m0 : 0;
    const uint32_t nst = (nm + MS - 1) / MS;     // stages of this task
    const size_t LN = (size_t)L * N;
    const uint64_t *xsrc = sg.X + (size_t)limb * N + k0;   // input row r at xsrc + r*LN
    const uint64_t *wsrc = sg.W + (size_t)limb * N + k0;   // weight poly j at wsrc + j*LN
    const int tid = threadIdx.x;
    const uint32_t g0 = ring.gi;

    // channels m0 + i*MS ... into ring slot (g0 + i) % kMacStages, once every warp has
    // handed its last use back; false: that wait ran out
    auto issue_w = [&](uint32_t i) {
        const uint32_t n = g0 + i, st = n % kMacStages, c0 = m0 + i * MS;
        if (n >= (uint32_t)kMacStages) {
            if (!mbar_wait(&bars[1 + kMacStages + st], (n / kMacStages - 1) & 1)) return false;
            fence_proxy_async();
        }
        const uint32_t nr = min(MS, m1 - c0) * G;
        mbar_arrive_expect_tx(&bars[1 + st], nr * ROW_BYTES);
        const uint64_t *src = wsrc + (size_t)c0 * G * LN;
        uint64_t *dst = ws + (size_t)st * SR * KC;
        const uint64_t pol = l2_evict_first_policy();  // each weight slot is read once per layer
        for (uint32_t r = 0; r < nr; ++r) bulk_g2s_stream(dst + (size_t)r * KC, src + r * LN, ROW_BYTES, &bars[1 + st], pol);
        return true;
    };
    uint32_t issued = 0;  // thread 0: stages of this task issued
    bool ok = true;
    if (tid == 0) {
        fence_proxy_async();  // earlier generic accesses to this shared memory before the copies
        mbar_arrive_expect_tx(&bars[0], rows * ROW_BYTES);
        for (uint32_t r = 0; r < rows; ++r) bulk_g2s(xs + (size_t)r * KC, xsrc + r * LN, ROW_BYTES, &bars[0]);
        while (ok && issued < (uint32_t)kMacStages && issued < nst) {
            ok = issue_w(issued);
            if (ok) ++issued;
        }
    }

    const LimbConst &lc = sg.limbs[limb];
    const uint64_t q = lc.q, nq = 0ull - q, r64 = lc.r64, r64_s = lc.r64_s;
    const uint32_t ones = (uint32_t)lc.one_s;
    // inputs and weights are canonical (< q < 2^50)
    const uint32_t sc = (uint32_t)lc.special_c;
    const bool special = sc != 0 && G <= kMacSpecialTerms;
    uint32_t p25, p28;
    asm("mov.u32 %0, 0x2000000;" : "=r"(p25));
    asm("mov.u32 %0, 0x10000000;" : "=r"(p28));
    const uint32_t k = tid % KC, h = tid / KC;  // h is warp-uniform
    const uint32_t xstep = P * KC;
    ok = mbar_wait(&bars[0], ring.xuse & 1) && ok;
    for (uint32_t e = tid; e < rows * KC; e += NT) xs[e] = split25(xs[e]);
    ok = __syncthreads_and(ok);
    const size_t chP = (size_t)P * LN;  // output words of a channel

    // CR channels x the two components of a block
    auto tile = [&](auto cr, const uint64_t *xp, const uint64_t *wk, uint64_t *yp) {
        constexpr int CR = decltype(cr)::value;
        MacAcc25 acc[CR][2];
#pragma unroll
        for (int c = 0; c < CR; ++c) {
            mac25_zero(acc[c][0]);
            mac25_zero(acc[c][1]);
        }
#pragma unroll 2
        for (uint32_t g = 0; g < G; ++g, xp += xstep, wk += KC) {
            uint64_t xv[2], wv[CR];
            uint32_t xt[2], wt[CR];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                xv[r] = xp[r * KC];
                xt[r] = (uint32_t)xv[r] + (uint32_t)(xv[r] >> 32);
            }
#pragma unroll
            for (int c = 0; c < CR; ++c) {
                wv[c] = split25(wk[(size_t)c * G * KC]);
                wt[c] = (uint32_t)wv[c] + (uint32_t)(wv[c] >> 32);
            }
#pragma unroll
            for (int c = 0; c < CR; ++c)
#pragma unroll
                for (int r = 0; r < 2; ++r) mac25_add(acc[c][r], xv[r], xt[r], wv[c], wt[c]);
        }
#pragma unroll
        for (int c = 0; c < CR; ++c)
#pragma unroll
            for (int r = 0; r < 2; ++r)
                yp[c * chP + r * LN] = special ? mac25_reduce_special(acc[c][r], q, sc, p25, p28)
                                               : mac25_reduce(acc[c][r], q, nq, r64, r64_s, ones);
    };
    using I1 = std::integral_constant<int, 1>;
    using I2 = std::integral_constant<int, 2>;
    const uint64_t *xk = xs + k;
    uint32_t job = h;  // this row group's next tile, counted from the stage's first
    for (uint32_t i = 0; ok && i < nst; ++i) {
        const uint32_t st = (g0 + i) % kMacStages;
        if (!__all_sync(0xffffffffu, mbar_wait(&bars[1 + st], ((g0 + i) / kMacStages) & 1))) {
            ok = false;
            break;
        }
        const uint32_t c0 = m0 + i * MS, cnt = min(MS, m1 - c0);
        const uint64_t *wst = ws + (size_t)st * SR * KC + k;
        uint64_t *yk = sg.Y + (size_t)limb * N + k0 + k + c0 * chP;
        const uint32_t jobs = (cnt + 1) / 2 * B;  // (channel pair, block), block fastest
        uint32_t cp = job / B, b = job - cp * B;
        for (; job < jobs; job += H) {
            const uint64_t *xp = xk + 2 * b * KC, *wk = wst + (size_t)2 * cp * G * KC;
            uint64_t *yp = yk + 2 * cp * chP + 2 * b * LN;
            if (2 * cp + 1 < cnt)
                tile(I2{}, xp, wk, yp);
            else
                tile(I1{}, xp, wk, yp);
            for (b += H; b >= B; b -= B) ++cp;
        }
        job -= jobs;
        __syncwarp();
        if ((tid & 31) == 0) mbar_arrive(&bars[1 + kMacStages + st]);  // this warp is done with the stage
        if (tid == 0 && issued < nst && issued < i + kMacStages) {
            ok = issue_w(issued);
            if (ok) ++issued;
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
    }
    ok = __syncthreads_and(ok);
    if (!ok) {
        if (tid == 0) {
            atomicExch(err, 2);
            // drain this task's bulk copies still in flight before the shared memory is reused
            mbar_wait(&bars[0], ring.xuse & 1);
            for (uint32_t j = issued > (uint32_t)kMacStages ? issued - kMacStages : 0; j < issued; ++j)
                mbar_wait(&bars[1 + (g0 + j) % kMacStages], ((g0 + j) / kMacStages) & 1);
        }
        return false;
    }
    ring.gi = g0 + nst;
    ring.xuse += 1;
    return true;
}

// The same sums as one CTA task of NT threads without staging: the input chunk in shared
// memory, cut at 2^25, and the weights straight from memory into registers, coalesced (32
// slots of a row per warp and load), four terms of a tile's loads in flight.  A row group
// waits for nobody, so a layer with few terms a sum is bound by memory.  Thread (k, h) owns
// slot k0 + k; the H row groups take tiles of CR channels x RR of the P = 2B rows in turn
// (RR divides P, rows fastest), CR*RR = 4 sums (24 registers, so that 32 warps fit an SM).
// Each weight is loaded once per RR rows, from memory once and then from the caches.
// Measured on GB300, the whole layer with its transforms: 256 -> 256 channels at N = 16384
// (G = 4, B = 1, 802 MB in and out of this task) 545 us through the ring, 459 streamed, of
// which this task is 165 us, 72 % of measured copy bandwidth; 2048 -> 1000 classifier
// (G = 24, B = 1) 88 -> 76 us; 16 -> 64 channels 55x55 (B = 2) 112 -> 103 us;
// 64 -> 64 channels 56x56 (G = 8, B = 4, through the ring 107 us for this task) 227 -> 207 us.
template <int KC, int NT, int CR, int RR>
__device__ __forceinline__ void mac_stream_task(const MacSeg &sg, uint32_t chunk, uint32_t limb, uint32_t m0,
                                                uint32_t m1, uint64_t *xs)
{
    constexpr uint32_t H = NT / KC;
    static_assert(NT % KC == 0 && KC % 32 == 0, "whole warps per row group");
    const uint32_t G = sg.G, P = 2 * sg.B, rows = G * P;
    const size_t LN = (size_t)sg.L * sg.N, off = (size_t)limb * sg.N + chunk * KC;
    const uint32_t k = threadIdx.x % KC, h = threadIdx.x / KC;
    const uint64_t *xg = after_wait(sg.X + off + k);
    for (uint32_t r = h; r < rows; r += H) xs[r * KC + k] = split25(ld_data(xg + r * LN));
    const LimbConst &lc = sg.limbs[limb];
    const uint64_t q = lc.q;
    const uint32_t sc = (uint32_t)lc.special_c;
    const bool special = sc != 0 && G <= kMacSpecialTerms;
    uint32_t p25, p28;
    asm("mov.u32 %0, 0x2000000;" : "=r"(p25));
    asm("mov.u32 %0, 0x10000000;" : "=r"(p28));
    __syncthreads();
    const size_t GLN = G * LN;
    const uint64_t *wk = sg.W + off + k;
    uint64_t *yk = sg.Y + off + k;
    auto tile = [&](auto cr, uint32_t m, uint32_t r0) {
        constexpr int CN = decltype(cr)::value;
        const uint64_t *w = wk + m * GLN, *xp = xs + r0 * KC + k;
        MacAcc25 acc[CN][RR];
#pragma unroll
        for (int c = 0; c < CN; ++c)
#pragma unroll
            for (int r = 0; r < RR; ++r) mac25_zero(acc[c][r]);
        auto terms = [&](auto ng) {  // ng channel groups, their weights loaded first
            constexpr int NG = decltype(ng)::value;
            uint64_t wv[NG][CN];
#pragma unroll
            for (int g = 0; g < NG; ++g, w += LN)
#pragma unroll
                for (int c = 0; c < CN; ++c) wv[g][c] = ld_near(w + c * GLN);
#pragma unroll
            for (int g = 0; g < NG; ++g, xp += P * KC) {
                uint32_t wt[CN];
#pragma unroll
                for (int c = 0; c < CN; ++c) {
                    wv[g][c] = split25(wv[g][c]);
                    wt[c] = (uint32_t)wv[g][c] + (uint32_t)(wv[g][c] >> 32);
                }
#pragma unroll
                for (int r = 0; r < RR; ++r) {
                    const uint64_t xv = xp[r * KC];
                    const uint32_t xt = (uint32_t)xv + (uint32_t)(xv >> 32);
#pragma unroll
                    for (int c = 0; c < CN; ++c) mac25_add(acc[c][r], xv, xt, wv[g][c], wt[c]);
                }
            }
        };
        uint32_t g = 0;
        for (; g + 4 <= G; g += 4) terms(std::integral_constant<int, 4>{});
        for (; g < G; ++g) terms(std::integral_constant<int, 1>{});
#pragma unroll
        for (int c = 0; c < CN; ++c)
#pragma unroll
            for (int r = 0; r < RR; ++r)
                yk[((size_t)(m + c) * P + r0 + r) * LN] =
                    special ? mac25_reduce_special(acc[c][r], q, sc, p25, p28)
                            : mac25_reduce(acc[c][r], q, 0ull - q, lc.r64, lc.r64_s, (uint32_t)lc.one_s);
    };
    const uint32_t tiles = P / RR;  // of a channel
    uint32_t m = m0 + h / tiles * CR, t = h % tiles;
    while (m < m1) {
        if (CR == 1 || m + CR <= m1)
            tile(std::integral_constant<int, CR>{}, m, t * RR);
        else
            tile(std::integral_constant<int, 1>{}, m, t * RR);
        for (t += H; t >= tiles; t -= tiles) m += CR;
    }
}

}  // namespace hc
