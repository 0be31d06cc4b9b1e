// hc_rotate.cu -- slot rotations of RLWE ciphertexts and the
// multiply-accumulate-rotate iteration of HELiKs-style linear layers over Z_P
// (SecONNds-P, Sec. 6.1: each iteration multiplies the input ciphertext by an
// NTT-preprocessed weight plaintext, accumulates, and rotates the accumulator
// by one slot; Sec. 2.1: rotations need a key-switching step with public
// evaluation keys).
//
// A rotation is the Galois automorphism sigma_g (X -> X^g) followed by key
// switching with one special prime p_sp and one digit per ciphertext limb:
//   d = sigma_g(c1);  D_j = d mod q_j lifted to every modulus of Q*p_sp;
//   (u0, u1) = sum_j NTT(D_j) . k_j over Q*p_sp, back to coefficients;
//   v = (u - [u]_{p_sp}) / p_sp over Q, [.] the centered residue;
//   out = (sigma_g(c0) + v0, v1).
// The key k_j = (b_j, a_j), b_j = -a_j s + e_j + p_sp * Qh_j [Qh_j^-1]_{q_j} sigma_g(s)
// (Qh_j = Q / q_j), comes from the secret-key holder; the GPU keeps it in the
// NTT domain over Q*p_sp.
#include <algorithm>
#include <new>
#include <vector>

#include "hc_arith.cuh"
#include "hc_async.cuh"
#include "hc_internal.h"

// per ciphertext limb i: p_sp mod q_i, p_sp^-1 mod q_i with its Shoup companion
struct ModDown {
    uint64_t p_mod_q, pinv, pinv_s;
};

struct hc_galois_key {
    uint32_t magic;
    const hc_ctx *ctx;     // ciphertext context: q_0 .. q_{L-1}
    hc_ctx *qp;            // owned: q_0 .. q_{L-1}, p_sp
    int device;
    uint32_t g;            // Galois element
    uint64_t special;
    uint64_t *d_key;       // [L][2][L+1][N], NTT domain over Q*p_sp
    ModDown *d_md;         // [L]
};

namespace hc {
namespace {

__device__ __forceinline__ uint64_t negmod(uint64_t v, uint64_t q) { return v ? q - v : 0; }

__device__ __forceinline__ uint64_t reduce_any(uint64_t v, const LimbConst &lc)
{
    return canon3(reduce_lazy(v, (uint32_t)lc.one_s, 0ull - lc.q), lc.q);
}

// The elementwise half of a rotation: division by p_sp, the sums, and the permutation the
// next key switch wants its input in.  With a = sigma(c) of the ciphertext c being rotated
// (already permuted),
//   w[ct][comp][i] = (comp == 0 ? a[ct][0][i] : 0) + (u_i - [u_sp]) / p_sp  (+ add) mod q_i
// is the rotated ciphertext, and out = sigma_g(w): coefficient k goes to k*g mod 2N, negated
// past N (g = 1: as it stands).  DIVIDE false: w = a, both components.  Reads are 16-byte
// and coalesced; the permutation is on the stores, each word stored once, where gathering
// it in the key switch would read every word L+1 times in 32-byte sectors.
// a's ciphertexts lie a_ct ciphertexts apart, add's add_ct.  ODD: a is a caller's buffer on an odd
// word, read word by word (chosen on the host: a test per load takes 2 us of 15 steps' 261).
// 2-D grid: y walks the rows (one polynomial limb each), x the N / 2 pairs of coefficients.
constexpr uint32_t kKsBlock = 128;

template <bool DIVIDE, bool ODD>
__global__ void __launch_bounds__(kKsBlock)
k_ks_apply(const uint64_t *a, const uint64_t *u, const uint64_t *add, uint64_t *out,
           const LimbConst *__restrict__ lq, const ModDown *__restrict__ md, uint64_t special, uint32_t L, uint32_t N,
           uint32_t g, uint32_t rows, uint32_t a_ct, uint32_t add_ct)
{
    pdl_begin();
    a = after_wait(a);
    u = after_wait(u);
    add = after_wait(add);
    const uint32_t k = 2 * (blockIdx.x * kKsBlock + threadIdx.x);
    const uint32_t mask2 = 2 * N - 1, L1 = L + 1;
    const uint64_t half = (special - 1) / 2;
    const uint32_t d0 = (uint32_t)((uint64_t)k * g) & mask2, d1 = (d0 + g) & mask2;
    for (uint32_t r = blockIdx.y; r < rows; r += gridDim.y) {
        const uint32_t cc = r / L, i = r - cc * L;  // cc = ct * 2 + comp
        const LimbConst &lc = lq[i];
        const uint64_t q = lc.q;
        auto strided = [&](uint32_t by) { return ((size_t)(cc >> 1) * by * 2 * L + (cc & 1) * L + i) * N + k; };
        auto ld2 = [](const uint64_t *p) { return ld_data(reinterpret_cast<const ulonglong2 *>(p)); };
        auto ld_a = [&](const uint64_t *p) {
            return !ODD ? ld2(p) : make_ulonglong2(ld_data(p), ld_data(p + 1));
        };
        ulonglong2 v;
        if constexpr (DIVIDE) {
            const ulonglong2 ui = ld2(u + ((size_t)cc * L1 + i) * N + k), us = ld2(u + ((size_t)cc * L1 + L) * N + k);
            const uint64_t pm = md[i].p_mod_q, pinv = md[i].pinv, pinv_s = md[i].pinv_s;
            auto div = [&](uint64_t x, uint64_t usp) {
                const uint64_t rsp = reduce_any(usp, lc);  // usp mod q_i
                // the centered residue: usp - p_sp when usp > (p_sp - 1) / 2
                const uint64_t cen = usp > half ? (rsp >= pm ? rsp - pm : rsp + q - pm) : rsp;
                const uint64_t diff = x >= cen ? x - cen : x + q - cen;
                return canon4(shoup_lazy(diff, pinv, pinv_s, 0ull - q), q);
            };
            if (add) {
                const ulonglong2 b = ld2(add + strided(add_ct));
                v.x = csub(div(ui.x, us.x) + b.x, q);
                v.y = csub(div(ui.y, us.y) + b.y, q);
            } else {
                v.x = div(ui.x, us.x);
                v.y = div(ui.y, us.y);
            }
            if (!(cc & 1)) {
                const ulonglong2 b = ld_a(a + (size_t)r * N + k);
                v.x = csub(v.x + b.x, q);
                v.y = csub(v.y + b.y, q);
            }
        } else {
            v = ld_a(a + strided(a_ct));
        }
        uint64_t *o = out + (size_t)r * N;
        if (g == 1 && ((uintptr_t)out & 15) == 0) {
            *reinterpret_cast<ulonglong2 *>(o + k) = v;
        } else {
            o[d0 & (N - 1)] = d0 < N ? v.x : negmod(v.x, q);
            o[d1 & (N - 1)] = d1 < N ? v.y : negmod(v.y, q);
        }
    }
}

// term list of a batch of products: output o = m*B + b sums the G terms (input g*B + b,
// plaintext m*G + g)
__global__ void k_product_terms(uint32_t *term_ptr, uint32_t *terms, uint32_t G, uint32_t B, uint32_t n_out)
{
    for (uint32_t o = blockIdx.x * blockDim.x + threadIdx.x; o <= n_out; o += gridDim.x * blockDim.x) {
        term_ptr[o] = o * G;
        if (o < n_out) {
            const uint32_t m = o / B, b = o % B;
            for (uint32_t g = 0; g < G; ++g) {
                terms[2 * (o * G + g)] = g * B + b;
                terms[2 * (o * G + g) + 1] = m * G + g;
            }
        }
    }
}

struct Buf {
    void *p = nullptr;
    cudaStream_t s;
    explicit Buf(cudaStream_t st) : s(st) {}
    ~Buf() { dev_free(p, s); }
};

bool key_ok(const hc_galois_key *k) { return k && k->magic == kMagicGaloisKey; }

// Device scratch of the rotations of n ciphertexts: one permuted ciphertext buffer and the key
// switch's result.
struct RotateScratch {
    Buf mem;
    uint64_t *a, *u;
    explicit RotateScratch(cudaStream_t s) : mem(s) {}
    hc_status alloc(const hc_ctx *ctx, size_t n, cudaStream_t s)
    {
        const size_t ct = n * 2 * ctx->L * (size_t)ctx->N, ks = n * 2 * (ctx->L + 1) * (size_t)ctx->N;
        if (n * 2 * (ctx->L + 1) > 0xffffffffu) return set_error(HC_ERR_INVALID_ARG, "batch too large");
        mem.p = dev_alloc((ct + ks) * 8, s);
        if (!mem.p) return set_error(HC_ERR_OOM, "scratch allocation failed");
        a = (uint64_t *)mem.p;
        u = a + ct;
        return HC_OK;
    }
};

// out[m*B + b] = INTT(sum_g x[g*B + b] . w[m*G + g]), x forward transformed.  The blocked
// MAC reads each weight once and sums at the multiply pipe's rate, and the inverse
// transforms run as a launch of their own; k_mac_intt, which reads its terms pair by pair
// from each output's CTA and stores word by word, stays for what does not fit and for an
// output on an odd word.  Measured on GB300,
// N = 8192, L = 3: a layer of 288 outputs of 16 terms and its rotations 1011 us with
// k_mac_intt (376 us of it), 929 so; an iteration of 16 products 281 and 271 us.
hc_status products(const hc_ctx *ctx, const uint64_t *x, const uint64_t *w, uint32_t G, uint32_t B, uint32_t M,
                   uint64_t *out, cudaStream_t s)
{
    const uint32_t n_out = M * B;
    if (mac_conv_fits(G, B) && !odd_word(out)) {
        const hc_status st = launch_mac_conv(ctx, x, w, out, G, B, M, s);
        return st == HC_OK ? launch_ntt_inv_ct(ctx, out, out, n_out, s) : st;
    }
    Buf tmp(s);
    tmp.p = dev_alloc(((size_t)n_out + 1 + 2 * (size_t)n_out * G) * sizeof(uint32_t), s);
    if (!tmp.p) return set_error(HC_ERR_OOM, "scratch allocation failed");
    uint32_t *term_ptr = (uint32_t *)tmp.p, *terms = term_ptr + n_out + 1;
    k_product_terms<<<(n_out + 256) / 256, 256, 0, s>>>(term_ptr, terms, G, B, n_out);
    HC_CUDA_TRY(cudaGetLastError());
    return launch_mac_intt(ctx, x, w, MacTerms{term_ptr, terms}, out, n_out, s);
}

// out = sigma_g(a), or with u = sigma_g of the rotation that a, u (+ add) finish
hc_status ks_apply(const hc_ctx *ctx, const hc_galois_key *key, const uint64_t *a, const uint64_t *u,
                   const uint64_t *add, uint64_t *out, uint32_t g, size_t n, cudaStream_t s, uint32_t a_ct = 1,
                   uint32_t add_ct = 1)
{
    const uint32_t rows = (uint32_t)(n * 2 * ctx->L);
    ProfileScope ps("k_ks_apply", s);
    const cudaError_t e = launch_programmatic(
        odd_word(a) ? (u ? k_ks_apply<true, true> : k_ks_apply<false, true>)
                    : (u ? k_ks_apply<true, false> : k_ks_apply<false, false>),
        dim3(ctx->N / 2 / kKsBlock, rows < 65535 ? rows : 65535), dim3(kKsBlock), 0, s, true, a, u, add, out,
        ctx->d_limbs, key->d_md, key->special, ctx->L, ctx->N, g, rows, a_ct, add_ct);
    return e == cudaSuccess ? HC_OK : cuda_error(e, "launch k_ks_apply");
}

// u = key switch of the permuted ciphertexts a
hc_status ks_switch(const hc_galois_key *key, const uint64_t *a, uint64_t *u, size_t n, cudaStream_t s)
{
    const hc_ctx *qp = key->qp;
    const KsArgs args{a, key->d_key, u, qp->d_limbs, qp->L - 1};
    switch (qp->logN) {
    case 12: return qp->fold ? launch_ks_n<12, true>(args, n, qp->sms, s) : launch_ks_n<12, false>(args, n, qp->sms, s);
    case 13: return qp->fold ? launch_ks_n<13, true>(args, n, qp->sms, s) : launch_ks_n<13, false>(args, n, qp->sms, s);
    case 14: return qp->fold ? launch_ks_n<14, true>(args, n, qp->sms, s) : launch_ks_n<14, false>(args, n, qp->sms, s);
    default: return set_error(HC_ERR_UNSUPPORTED, "unsupported N = %u", qp->N);
    }
}

// acc = P_steps;  acc = rot_{key(i)}(acc) + P_i, i = steps-1 .. 0;  out = acc.  Ciphertext j
// of P_i is prods[i*by_i + j*by_j].  Each step is two launches: the key switch, then the
// division and the addition, whose stores are already permuted for the next step.  The
// accumulators a step reads lie in the scratch and in out in turn, the last step's in the
// scratch, so that a chain needs no more memory than one rotation.
template <class KeyAt>
hc_status rotate_chain(const hc_ctx *ctx, const KeyAt &key_at, const uint64_t *prods, uint32_t by_i,
                       uint32_t by_j, uint32_t steps, size_t n, uint64_t *out, cudaStream_t s)
{
    RotateScratch sc(s);
    hc_status st = sc.alloc(ctx, n, s);
    if (st != HC_OK) return st;
    auto acc = [&](uint32_t i) { return i & 1 ? out : sc.a; };
    const size_t step = (size_t)by_i * 2 * ctx->L * ctx->N;
    const hc_galois_key *key = key_at(steps - 1);
    st = ks_apply(ctx, key, prods + steps * step, nullptr, nullptr, acc(steps - 1), key->g, n, s, by_j);
    for (uint32_t i = steps; st == HC_OK && i-- > 0;) {
        st = ks_switch(key, acc(i), sc.u, n, s);
        if (st != HC_OK) break;
        const hc_galois_key *next = i ? key_at(i - 1) : nullptr;
        st = ks_apply(ctx, key, acc(i), sc.u, prods + i * step, i ? acc(i - 1) : out, next ? next->g : 1, n, s, 1, by_j);
        key = next;
    }
    return st;
}

}  // namespace

void galois_key_destroy(hc_galois_key *k)
{
    DeviceGuard g(k->device);
    dev_free_persistent(k->d_key);
    dev_free_persistent(k->d_md);
    hc_free(k->qp);
    k->magic = kMagicDead;
    delete k;
}

}  // namespace hc

using namespace hc;

extern "C" {

hc_status hc_galois_key_create(const hc_ctx *ctx, uint64_t special_prime, uint32_t galois_elt, const uint64_t *h_key,
                               hc_galois_key **out, void *cuda_stream)
{
    if (!out) return set_error(HC_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!ctx || ctx->magic != kMagicCtx) return set_error(HC_ERR_INVALID_ARG, "invalid context");
    if (!h_key) return set_error(HC_ERR_INVALID_ARG, "h_key is NULL");
    const uint32_t L = ctx->L, N = ctx->N;
    if (L + 1 > kMaxLimbs) return set_error(HC_ERR_INVALID_ARG, "no room for the special prime (L = %u)", L);
    if (!(galois_elt & 1) || galois_elt >= 2 * N)
        return set_error(HC_ERR_INVALID_ARG, "Galois element must be odd and below 2N (got %u)", galois_elt);
    for (uint32_t i = 0; i < L; ++i)
        if (ctx->q[i] == special_prime) return set_error(HC_ERR_BAD_MODULUS, "special prime equals q[%u]", i);
    DeviceGuard dg(ctx->device);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    uint64_t moduli[kMaxLimbs];
    for (uint32_t i = 0; i < L; ++i) moduli[i] = ctx->q[i];
    moduli[L] = special_prime;
    hc_ctx *qp = nullptr;
    hc_status st = hc_ctx_create_ex(N, moduli, L + 1, ctx->t, 0, &qp);  // validates the special prime
    if (st != HC_OK) return st;
    hc_galois_key *k = new (std::nothrow) hc_galois_key();
    if (!k) {
        hc_free(qp);
        return set_error(HC_ERR_OOM, "host allocation failed");
    }
    k->magic = kMagicGaloisKey;
    k->ctx = ctx;
    k->qp = qp;
    k->device = ctx->device;
    k->g = galois_elt;
    k->special = special_prime;
    std::vector<ModDown> md(L);
    for (uint32_t i = 0; i < L; ++i) {
        const uint64_t q = ctx->q[i];
        md[i].p_mod_q = special_prime % q;
        md[i].pinv = powmod_u64(md[i].p_mod_q, q - 2, q);
        md[i].pinv_s = shoup_companion(md[i].pinv, q);
    }
    const size_t key_words = (size_t)L * 2 * (L + 1) * N;
    k->d_key = (uint64_t *)dev_alloc_persistent(key_words * 8);
    k->d_md = (ModDown *)dev_alloc_persistent(L * sizeof(ModDown));
    if (!k->d_key || !k->d_md) {
        galois_key_destroy(k);
        return set_error(HC_ERR_OOM, "device allocation of the Galois key failed");
    }
    cudaError_t e = cudaMemcpy(k->d_key, h_key, key_words * 8, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(k->d_md, md.data(), L * sizeof(ModDown), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        galois_key_destroy(k);
        return cuda_error(e, "uploading the Galois key");
    }
    st = check_inputs(qp, k->d_key, (size_t)2 * L, s);
    if (st == HC_OK) st = launch_ntt_fwd(qp, k->d_key, k->d_key, (size_t)2 * L, s);
    if (st == HC_OK) {
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = cuda_error(e, "Galois key preprocessing");
    }
    if (st != HC_OK) {
        galois_key_destroy(k);
        return st;
    }
    *out = k;
    return HC_OK;
}

hc_status hc_ct_rotate(const hc_ctx *ctx, const hc_galois_key *key, const uint64_t *d_ct_in, uint64_t *d_ct_out,
                       size_t n_ct, void *cuda_stream)
{
    if (!ctx || ctx->magic != kMagicCtx || !key_ok(key)) return set_error(HC_ERR_INVALID_ARG, "invalid context or key");
    if (key->ctx != ctx) return set_error(HC_ERR_INVALID_ARG, "key was made for another context");
    if (n_ct == 0) return HC_OK;
    if (!d_ct_in || !d_ct_out) return set_error(HC_ERR_INVALID_ARG, "null ciphertext buffer");
    if (d_ct_in == d_ct_out) return set_error(HC_ERR_INVALID_ARG, "in place rotation is not supported");
    DeviceGuard dg(ctx->device);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    hc_status st = check_inputs(ctx, d_ct_in, 2 * n_ct, s);
    if (st != HC_OK) return st;
    RotateScratch sc(s);
    st = sc.alloc(ctx, n_ct, s);
    if (st == HC_OK) st = ks_apply(ctx, key, d_ct_in, nullptr, nullptr, sc.a, key->g, n_ct, s);
    if (st == HC_OK) st = ks_switch(key, sc.a, sc.u, n_ct, s);
    if (st == HC_OK) st = ks_apply(ctx, key, sc.a, sc.u, nullptr, d_ct_out, 1, n_ct, s);
    return st;
}

hc_status hc_mac_rotate_many(const hc_ctx *ctx, const hc_galois_key *key, const uint64_t *d_ct, uint32_t m,
                             const uint64_t *d_w_ntt, uint32_t n, uint64_t *d_out, void *cuda_stream)
{
    if (!ctx || ctx->magic != kMagicCtx || !key_ok(key)) return set_error(HC_ERR_INVALID_ARG, "invalid context or key");
    if (key->ctx != ctx) return set_error(HC_ERR_INVALID_ARG, "key was made for another context");
    if (!d_ct || !d_w_ntt || !d_out || n == 0 || m == 0) return set_error(HC_ERR_INVALID_ARG, "null buffer or empty batch");
    if ((uint64_t)n * m > 0x3fffffffu) return set_error(HC_ERR_INVALID_ARG, "batch too large");
    if (odd_word(d_w_ntt)) return set_error(HC_ERR_INVALID_ARG, "d_w_ntt is not aligned to 16 bytes");
    DeviceGuard dg(ctx->device);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    hc_status st = check_inputs(ctx, d_ct, (size_t)2 * m, s);
    if (st == HC_OK) st = check_inputs(ctx, d_w_ntt, n, s);
    if (st != HC_OK) return st;
    // The products x_j * w_i do not depend on the accumulators: all m*n run first, in
    // one batch (forward NTT of the x_j once, then the products and their inverse NTTs);
    // the chain then only rotates and adds, all m accumulators per step, the add fused
    // into the division kernel:
    //   P_i = x * w_i (m ciphertexts);  acc = P_{n-1};  acc = rot(acc) + P_i, i = n-2 .. 0.
    const uint32_t L = ctx->L, N = ctx->N;
    const size_t ct_words = (size_t)2 * L * N, mn = (size_t)m * n;
    Buf tmp(s);
    tmp.p = dev_alloc((mn + m) * ct_words * 8, s);
    if (!tmp.p) return set_error(HC_ERR_OOM, "scratch allocation failed");
    uint64_t *ctn = (uint64_t *)tmp.p, *prods = ctn + (size_t)m * ct_words;  // prods [n][m][2][L][N]
    st = launch_ntt_fwd(ctx, d_ct, ctn, (size_t)2 * m, s);
    if (st != HC_OK) return st;
    uint64_t *first = n == 1 ? d_out : prods;  // P_0 of a one-term iteration is the result
    st = products(ctx, ctn, d_w_ntt, 1, m, n, first, s);
    if (st != HC_OK || n == 1) return st;
    return rotate_chain(ctx, [&](uint32_t) { return key; }, prods, m, 1, n - 1, m, d_out, s);
}

hc_status hc_mac_rotate(const hc_ctx *ctx, const hc_galois_key *key, const uint64_t *d_ct, const uint64_t *d_w_ntt,
                        uint32_t n, uint64_t *d_out, void *cuda_stream)
{
    return hc_mac_rotate_many(ctx, key, d_ct, 1, d_w_ntt, n, d_out, cuda_stream);
}

hc_status hc_zp_plain_preprocess(const hc_ctx *ctx, uint64_t P, const uint64_t *h_plain, size_t n, uint64_t *d_out,
                                 void *cuda_stream)
{
    if (!ctx || ctx->magic != kMagicCtx) return set_error(HC_ERR_INVALID_ARG, "invalid context");
    if (n == 0) return HC_OK;
    if (!h_plain || !d_out) return set_error(HC_ERR_INVALID_ARG, "null buffer");
    if (P < 3 || P >= (1ull << 50)) return set_error(HC_ERR_INVALID_ARG, "plaintext modulus out of range");
    const uint32_t L = ctx->L, N = ctx->N;
    // centered lift of every coefficient into each q_i, on the host; NTT on the device
    std::vector<uint64_t> lifted(n * L * N);
    for (size_t p = 0; p < n; ++p)
        for (uint32_t k = 0; k < N; ++k) {
            const uint64_t v = h_plain[p * N + k];
            if (v >= P) return set_error(HC_ERR_RANGE, "plaintext coefficient %llu >= P", (unsigned long long)v);
            const bool neg = v > (P - 1) / 2;
            for (uint32_t i = 0; i < L; ++i) {
                const uint64_t q = ctx->q[i];
                lifted[(p * L + i) * N + k] = neg ? q - (P - v) % q : v % q;
            }
        }
    DeviceGuard dg(ctx->device);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    HC_CUDA_TRY(cudaMemcpyAsync(d_out, lifted.data(), lifted.size() * 8, cudaMemcpyHostToDevice, s));
    hc_status st = launch_ntt_fwd(ctx, d_out, d_out, n, s);
    if (st != HC_OK) return st;
    HC_CUDA_TRY(cudaStreamSynchronize(s));  // the host copy must outlive the upload
    return HC_OK;
}

hc_status hc_zp_conv(const hc_ctx *ctx, const hc_conv_desc *desc, const hc_galois_key *key_1,
                     const hc_galois_key *key_row, const uint64_t *d_w_ntt, const uint64_t *d_ct_in,
                     uint64_t *d_ct_out, void *cuda_stream)
{
    if (!ctx || ctx->magic != kMagicCtx) return set_error(HC_ERR_INVALID_ARG, "invalid context");
    if (!desc || !d_w_ntt || !d_ct_in || !d_ct_out) return set_error(HC_ERR_INVALID_ARG, "null descriptor or buffer");
    ZpConvGeom g;
    hc_status st = zp_conv_geometry(desc, ctx->N, &g);
    if (st != HC_OK) return st;
    const uint32_t L = ctx->L, N = ctx->N, C = desc->C, kk = desc->kh * desc->kw, Y = g.Y;
    // the two rotations of the iteration: by 1 slot within a kernel row, by Wp - kw + 1 to the next
    const uint32_t g1 = 5, grow = (uint32_t)powmod_u64(5, g.step_row, 2ull * N);
    if (desc->kw > 1 && (!key_ok(key_1) || key_1->ctx != ctx || key_1->g != g1))
        return set_error(HC_ERR_INVALID_ARG, "key_1 must be a Galois key of element 5 for this context");
    if (desc->kh > 1 && (!key_ok(key_row) || key_row->ctx != ctx || key_row->g != grow))
        return set_error(HC_ERR_INVALID_ARG, "key_row must be a Galois key of element 5^%u mod 2N = %u", g.step_row,
                         grow);
    const uint64_t n_out64 = (uint64_t)kk * Y;
    if (n_out64 * C > 0x3fffffffu) return set_error(HC_ERR_INVALID_ARG, "layer too large");
    if (odd_word(d_w_ntt)) return set_error(HC_ERR_INVALID_ARG, "d_w_ntt is not aligned to 16 bytes");
    const uint32_t n_out = (uint32_t)n_out64;
    DeviceGuard dg(ctx->device);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    st = check_inputs(ctx, d_ct_in, (size_t)2 * C, s);
    if (st != HC_OK) return st;
    // P_{y,i} = sum_c x_c * w_{y,i,c}: forward NTT of the C inputs once, then the products
    // and inverse NTTs of the kk*Y outputs (ordered [y][i], as the weights); the chain then
    // rotates and adds, all Y accumulators per step, the add
    // fused into the division's kernel:
    //   acc = P_{kk-1};  acc = rot^(step_i)(acc) + P_i, i = kk-2 .. 0.
    const size_t ct_words = (size_t)2 * L * N;
    const size_t prod_words = kk > 1 ? (size_t)n_out * ct_words : 0;
    Buf tmp(s);
    tmp.p = dev_alloc(((size_t)C * ct_words + prod_words) * 8, s);
    if (!tmp.p) return set_error(HC_ERR_OOM, "scratch allocation failed");
    uint64_t *ctn = (uint64_t *)tmp.p, *prods = ctn + (size_t)C * ct_words;  // prods [Y][kk][2][L][N]
    st = launch_ntt_fwd(ctx, d_ct_in, ctn, (size_t)2 * C, s);
    if (st != HC_OK) return st;
    st = products(ctx, ctn, d_w_ntt, C, 1, n_out, kk == 1 ? d_ct_out : prods, s);
    if (st != HC_OK || kk == 1) return st;
    // offsets i and i + 1 lie in one kernel row unless i + 1 starts a new one
    auto key_at = [&](uint32_t i) { return (i + 1) % desc->kw == 0 ? key_row : key_1; };
    return rotate_chain(ctx, key_at, prods, 1, kk, kk - 1, Y, d_ct_out, s);
}

}  // extern "C"
