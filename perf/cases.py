"""What the speed of this library is measured on: calls that a server of SecONNds' linear layers makes,
through the C ABI's Python binding, at sizes of the paper's networks (SqueezeNet-1.1, ResNet-50), of the
benchmark and of the tests.

  listed()             the cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  the inputs, contexts, weights, keys and plans a server holds before the call
  run(state)           one call and its outputs
  work(case)           bytes and operations the call cannot do without
  exact(case, seed)    the outputs from their definition, in torch's 64-bit integers, without the library

Every output is a canonical residue, so results are exact integers.
"""
import functools
import math

import numpy as np
import torch

from paper_2506_11586_gb300 import _lib as L
from paper_2506_11586_gb300.inputs import CANONICAL_PRIMES, RESNET50_FC, SQUEEZENET_1_1, T_PLAIN, uneven_mix

DEGREES = ((4096, 2), (8192, 3), (16384, 4))  # ring degree and limb count used together


# ------------------------------------------------------------------ cases ---

def _conv(name, N, nl, C, H, W, M, k, pad, **more):
    return dict(kind="conv", name=name, N=N, L=nl, bits=50, C=C, H=H, W=W, M=M, k=k, pad=pad, mode=0, form=0, **more)


def listed():
    return [
        # sixteen products with a slot of their own each: the smallest call
        dict(kind="ctpt", name="ctpt_16_n4096", N=4096, L=2, bits=50, n=16, n_out=16),
        # ResNet-50's classifier: few ciphertexts, latency counts
        dict(kind="fc", name="fc_2048x1000_n16384", N=16384, L=4, C=RESNET50_FC[0], M=RESNET50_FC[1]),
        # a 1x1 layer on a 13x13 map, SqueezeNet's most frequent size
        _conv("conv_fire6_squeeze", 8192, 3, 256, 13, 13, 48, 1, 0),
        # the benchmark's layer with the launch form its autotuner settles on
        dict(_conv("conv_56x56x64_chains", 8192, 3, 64, 56, 56, 64, 3, 1), form=2),
        # the same layer with its weights transformed by every call (online preprocessing), defaults otherwise
        dict(_conv("conv_56x56x64_online", 8192, 3, 64, 56, 56, 64, 3, 1), mode=1),
        # a wide 3x3 layer of ResNet-50 on a small map at the large ring degree
        _conv("conv_res4_conv2_n16384", 16384, 4, 256, 14, 14, 256, 3, 1),
        # the server's whole step around a layer: share added, outputs masked, only what the client needs returned
        dict(_conv("step_fire2_expand3x3", 8192, 3, 16, 55, 55, 64, 3, 1), kind="step"),
        # a layer on the client's host buffers, copies included
        dict(_conv("host_fire4_expand3x3", 8192, 3, 32, 27, 27, 128, 3, 1), kind="host"),
        # every stride-1 convolution of SqueezeNet-1.1 as one plan: the largest call
        dict(kind="net", name="plan_squeezenet", N=8192, L=3, first=0, count=len(SQUEEZENET_1_1)),
        # an uneven batch of standalone products, 40/40/20 % of the three degrees
        dict(kind="products", name="plan_products_2000", n=2000),
        # one client's multiply-accumulate-rotate iteration: a chain of 15 key-switched rotations
        dict(kind="macrot", name="mac_rotate_16", N=8192, L=3, n=16, m=1),
        # a convolution over Z_P by rotations of 32 ciphertexts at a time
        dict(kind="zpconv", name="zp_conv_fire2_expand3x3", N=8192, L=3, C=16, H=55, W=55, M=64, k=3, pad=1),
    ]


def _log(rng, lo, hi):
    return min(hi, int(lo * (hi / lo + 0.999 / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["ctpt", "fc", "conv", "conv", "conv", "step", "host", "net", "products", "macrot", "zpconv"])
    N, nl = rng.choice(DEGREES)
    if kind == "ctpt":
        n = _log(rng, 1, 64)
        return dict(kind=kind, N=N, L=rng.randint(1, 5), bits=rng.choice([50, 50, 45]), n=n, n_out=rng.choice([n, n, 1, max(1, n // 2)]))
    if kind == "fc":
        return dict(kind=kind, N=N, L=nl, C=_log(rng, 64, 2048), M=_log(rng, 10, 1000))
    if kind in ("conv", "step", "host"):
        while True:
            k = rng.choice([1, 3])
            H = _log(rng, 7, 56)
            c = dict(_conv("", N, nl, _log(rng, 3, 512), H, max(7, H - rng.randint(0, 3)), _log(rng, 8, 512), k, k // 2), kind=kind)
            if c["C"] * c["M"] * H * H <= 64 * 64 * 56 * 56 * (1 if kind == "host" else 4):
                break
        del c["name"]
        if kind == "conv":
            c.update(mode=rng.choice([0, 0, 0, 1]), form=rng.choice([0, 0, 2]), bits=rng.choice([50, 50, 50, 45]))
        return c
    if kind == "net":
        count = rng.randint(2, len(SQUEEZENET_1_1))
        return dict(kind=kind, N=N, L=nl, first=rng.randint(0, len(SQUEEZENET_1_1) - count), count=count if N < 16384 else min(count, 8))
    if kind == "products":
        return dict(kind=kind, n=_log(rng, 20, 2000))
    if kind == "macrot":
        return dict(kind=kind, N=N, L=nl, n=_log(rng, 2, 32), m=rng.choice([1, 1, 2, 5, 16]))
    side = _log(rng, 7, {4096: 40, 8192: 55, 16384: 55}[N])
    return dict(kind=kind, N=N, L=nl, C=_log(rng, 2, 16), H=side, W=side, M=_log(rng, 2, 64), k=3, pad=1)


# ----------------------------------------------------------------- inputs ---

def _is_prime(n):  # Miller-Rabin, deterministic below 3.3e24
    if n < 2:
        return False
    for p in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37):
        if n % p == 0:
            return n == p
    d, r = n - 1, 0
    while d % 2 == 0:
        d, r = d // 2, r + 1
    for a in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37):
        x = pow(a, d, n)
        if x in (1, n - 1):
            continue
        for _ in range(r - 1):
            x = x * x % n
            if x == n - 1:
                break
        else:
            return False
    return True


@functools.lru_cache(None)
def _primes(bits, n):
    """The n largest primes below 2^bits that are 1 mod 2^15, largest first."""
    out, q = [], (1 << bits) - (1 << 15) + 1
    while len(out) < n:
        if _is_prime(q):
            out.append(q)
        q -= 1 << 15
    return tuple(out)


def _moduli(case):
    return CANONICAL_PRIMES[:case["L"]] if case.get("bits", 50) == 50 else _primes(case["bits"], case["L"])


def _plain_prime():
    return _primes(37, 1)[0]


class _Rand:
    """Seeded uniform values, made on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def below(self, q, shape):
        return torch.randint(0, q, shape, dtype=torch.int64, device="cuda", generator=self.g)

    def residues(self, moduli, before, N):
        out = torch.empty(tuple(before) + (len(moduli), N), dtype=torch.int64, device="cuda")
        for i, q in enumerate(moduli):
            out[..., i, :] = self.below(q, tuple(before) + (N,))
        return out

    def int8(self, shape):
        return torch.randint(-128, 128, shape, dtype=torch.int8, device="cuda", generator=self.g).cpu().numpy()


def _empty(*shape):
    return torch.empty(shape, dtype=torch.int64, device="cuda")


def _special(moduli):
    return CANONICAL_PRIMES[len(moduli)]


def _host_words(t):
    return t.cpu().numpy().view(np.uint64)


def _net_shapes(case):
    return SQUEEZENET_1_1[case["first"]:case["first"] + case["count"]]


def _inputs(case, seed):
    """The random values of a case, in a fixed order; shared by prepare and exact."""
    r, kind, v = _Rand(seed), case["kind"], {}
    if kind == "ctpt":
        q = _moduli(case)
        v["ct"], v["pt"] = r.residues(q, (case["n"], 2), case["N"]), r.residues(q, (case["n"],), case["N"])
    elif kind == "fc":
        v["K"] = r.int8((case["M"], case["C"]))
        v["ct"] = r.residues(_moduli(case), (_fc_part(case["C"], case["M"], case["N"])[2], 2), case["N"])
    elif kind in ("conv", "step", "host"):
        k, p = case["k"], _part(case["C"], case["H"], case["W"], case["M"], case["k"], case["pad"], case["N"])
        v["K"] = r.int8((case["M"], case["C"], k, k))
        v["ct"] = r.residues(_moduli(case), (p["I"], 2), case["N"])
        if kind == "step":
            ho, wo = case["H"] + 2 * case["pad"] - k + 1, case["W"] + 2 * case["pad"] - k + 1
            v["share"], v["mask"] = r.below(T_PLAIN, (case["C"], case["H"], case["W"])), r.below(T_PLAIN, (case["M"], ho, wo))
    elif kind == "net":
        v["layers"] = []
        for s in _net_shapes(case):
            p = _part(s.C, s.H, s.W, s.M, s.kh, s.pad, case["N"])
            v["layers"].append((s, p, r.int8((s.M, s.C, s.kh, s.kw)), r.residues(_moduli(case), (p["I"], 2), case["N"])))
    elif kind == "products":
        lab = uneven_mix(case["n"], 3)
        v["classes"] = [(N, CANONICAL_PRIMES[:nl], int((lab == i).sum())) for i, (N, nl) in enumerate(DEGREES)]
        v["classes"] = [(N, q, r.residues(q, (n, 2), N), r.residues(q, (n,), N)) for N, q, n in v["classes"] if n]
    else:
        q, N = _moduli(case), case["N"]
        qp = q + (_special(q),)
        v["key"] = [r.residues(qp, (len(q), 2), N) for _ in range(1 if kind == "macrot" else 2)]
        if kind == "macrot":
            v["ct"], v["w"] = r.residues(q, (case["m"], 2), N), r.residues(q, (case["n"],), N)
        else:
            v["ct"], v["K"] = r.residues(q, (case["C"], 2), N), r.below(_plain_prime(), (case["M"], case["C"], case["k"], case["k"]))
    return v


def prepare(case, seed):
    kind, v = case["kind"], _inputs(case, seed)
    if kind == "products":
        items, outs, keep = [], [], []
        for N, q, ct, pt in v["classes"]:
            ctx, out = L.hc_ctx_create(N, q, T_PLAIN), torch.empty_like(ct)
            items.append(L.work_products(ctx, ct, pt, out))
            outs.append(out)
        return dict(kind=kind, plan=L.hc_plan_create(items), out=outs)
    q, N = _moduli(case), case["N"]
    ctx = L.hc_ctx_create(N, q, T_PLAIN)
    st = dict(kind=kind, ctx=ctx, **v)
    if kind == "ctpt":
        st["slots"] = np.arange(case["n"], dtype=np.uint32) % case["n_out"]
        st["out"] = _empty(case["n_out"], 2, len(q), N)
    elif kind == "fc":
        st["w"] = L.hc_weights_preprocess_fc(ctx, L.make_fc_desc(case["C"], case["M"]), v["K"])
        st["out"] = _empty(st["w"].O, 2, len(q), N)
    elif kind in ("conv", "step", "host"):
        desc = L.make_desc(case["C"], case["H"], case["W"], case["M"], case["k"], case["k"], case["pad"])
        L.hc_ctx_set_variant(ctx, L.KIND_CONV_FORM, case["form"])
        st["w"] = w = L.hc_weights_preprocess_ex(ctx, desc, v["K"], case["mode"])
        if kind == "step":
            st["c1"], st["slots"] = _empty(w.O, len(q), N), _empty(w.O, len(q), w.n_slots)
        elif kind == "host":
            st["ct"] = v["ct"].cpu().pin_memory()
            st["out"] = torch.empty((w.O, 2, len(q), N), dtype=torch.int64).pin_memory()
        else:
            st["out"] = _empty(w.O, 2, len(q), N)
    elif kind == "net":
        items, st["out"] = [], []
        for s, p, K, ct in st.pop("layers"):
            w = L.hc_weights_preprocess(ctx, L.make_desc(s.C, s.H, s.W, s.M, s.kh, s.kw, s.pad), K)
            st["out"].append(_empty(w.O, 2, len(q), N))
            items.append(L.work_conv(ctx, w, ct, st["out"][-1]))
        st["plan"] = L.hc_plan_create(items)
    elif kind == "macrot":
        st["key"] = L.hc_galois_key_create(ctx, _special(q), 5, _host_words(v["key"][0]))
        st["out"] = torch.empty_like(v["ct"])
    else:
        P = _plain_prime()
        ctx_p = L.hc_ctx_create(N, (P,), P)
        st["desc"] = desc = L.make_desc(case["C"], case["H"], case["W"], case["M"], case["k"], case["k"], case["pad"])
        step = case["W"] + 2 * case["pad"] - case["k"] + 1
        st["key"] = [L.hc_galois_key_create(ctx, _special(q), g, _host_words(t))
                     for g, t in zip((5, pow(5, step, 2 * N)), v["key"])]
        Y = (case["M"] + 1) // 2
        st["w"] = _empty(Y * case["k"] ** 2 * case["C"], len(q), N)
        L.hc_zp_conv_preprocess(ctx, ctx_p, desc, _host_words(v["K"]), st["w"])
        st["out"] = _empty(Y, 2, len(q), N)
    torch.cuda.synchronize()
    return st


def run(st):
    kind = st["kind"]
    if kind == "ctpt":
        L.hc_ctpt_mac(st["ctx"], st["ct"], st["pt"], st["slots"], st["out"])
    elif kind in ("net", "products"):
        L.hc_plan_run(st["plan"])
    elif kind == "step":
        L.hc_conv_server_step_sparse(st["ctx"], st["w"], st["ct"], st["share"], st["mask"], st["c1"], st["slots"])
        return [st["c1"], st["slots"]]
    elif kind == "host":
        L.hc_conv_ct_pt_host(st["ctx"], st["w"], st["ct"], st["out"])
    elif kind == "macrot":
        L.hc_mac_rotate_many(st["ctx"], st["key"], st["ct"], st["w"], st["out"])
    elif kind == "zpconv":
        L.hc_zp_conv(st["ctx"], st["desc"], st["key"][0], st["key"][1], st["w"], st["ct"], st["out"])
    else:
        L.hc_conv_ct_pt(st["ctx"], st["w"], st["ct"], st["out"])
    return st["out"]


# ------------------------------------------------------------------- work ---

def _ceil(a, b):
    return -(-a // b)


@functools.lru_cache(None)
def _part(C, H, W, M, k, pad, N):
    """The canonical partition of include/hconv.h: fewest polynomials 2I + P + 2O, then the largest
    block, then the most channels, then the widest block."""
    Hp, Wp, best = H + 2 * pad, W + 2 * pad, None
    for Hw in range(k, Hp + 1):
        for Ww in range(k, Wp + 1):
            if Hw * Ww > N:
                break
            Cw = min(C, N // (Hw * Ww))
            G, Bh, Bw = _ceil(C, Cw), _ceil(Hp - k + 1, Hw - k + 1), _ceil(Wp - k + 1, Ww - k + 1)
            B = Bh * Bw
            key = (2 * G * B + M * G + 2 * M * B, -Hw * Ww, -Cw, -Ww)
            if best is None or key < best[0]:
                best = (key, dict(Cw=Cw, Hw=Hw, Ww=Ww, G=G, B=B, Bw=Bw, I=G * B, P=M * G, O=M * B))
    return best[1]


@functools.lru_cache(None)
def _fc_part(C, M, N):
    """Canonical partition of a fully connected layer: (Cw, No, G, Mp)."""
    best = None
    for Cw in range(1, min(C, N) + 1):
        G = _ceil(C, Cw)
        No = min(M, N // Cw)
        Mp = _ceil(M, No)
        key = (2 * G + Mp * G + 2 * Mp, Mp * G, -Cw, _ceil(M, Mp))
        if best is None or key < best[0]:
            best = (key, (Cw, _ceil(M, Mp), G, Mp))
    return best[1]


def _ntt_mults(N):
    return N // 2 * int(math.log2(N))


def _rot_work(N, nl, n):
    """Words moved and modular products of rotating n ciphertexts (digits, key switch, division)."""
    limbs = nl * (nl + 1) + 2 * (nl + 1)
    return 4 * nl * N * n, n * (limbs * _ntt_mults(N) + 2 * nl * (nl + 1) * N + 2 * nl * N)


def _layer_work(N, nl, I, P, O, prods, online=False):
    return (nl * N * (2 * I + P + 2 * O),
            nl * ((2 * I + 2 * O + (P if online else 0)) * _ntt_mults(N) + 2 * prods * N))


def work(case):
    """Every input and weight word read once, every output word written once; a modular product with its
    addition counts as two operations."""
    kind, N, nl = case["kind"], case.get("N"), case.get("L")
    if kind == "ctpt":
        w = nl * N * (3 * case["n"] + 2 * case["n_out"])
        m = nl * ((2 * case["n"] + 2 * case["n_out"]) * _ntt_mults(N) + 2 * case["n"] * N)
    elif kind == "fc":
        Cw, No, G, Mp = _fc_part(case["C"], case["M"], N)
        w, m = _layer_work(N, nl, G, Mp * G, Mp, Mp * G)
    elif kind in ("conv", "step", "host"):
        p = _part(case["C"], case["H"], case["W"], case["M"], case["k"], case["pad"], N)
        w, m = _layer_work(N, nl, p["I"], p["P"], p["O"], case["M"] * p["I"], case["mode"] == 1)
        if kind == "step":
            w += nl * p["O"] * ((p["Hw"] - case["k"] + 1) * (p["Ww"] - case["k"] + 1) - N) + case["C"] * case["H"] * case["W"] \
                + case["M"] * (case["H"] + 2 * case["pad"] - case["k"] + 1) * (case["W"] + 2 * case["pad"] - case["k"] + 1)
    elif kind == "net":
        w = m = 0
        for s in _net_shapes(case):
            p = _part(s.C, s.H, s.W, s.M, s.kh, s.pad, N)
            a, b = _layer_work(N, nl, p["I"], p["P"], p["O"], s.M * p["I"])
            w, m = w + a, m + b
    elif kind == "products":
        lab, w, m = uneven_mix(case["n"], 3), 0, 0
        for i, (N, nl) in enumerate(DEGREES):
            n = int((lab == i).sum())
            w, m = w + 5 * nl * N * n, m + n * nl * (4 * _ntt_mults(N) + 2 * N)
    elif kind == "macrot":
        n, mm = case["n"], case["m"]
        w, m = _rot_work(N, nl, mm * (n - 1))
        w = nl * N * (4 * mm + n) + 2 * nl * (nl + 1) * N
        m += nl * (2 * mm * (1 + n) * _ntt_mults(N) + 2 * mm * n * N)
    else:
        Y, kk, C = (case["M"] + 1) // 2, case["k"] ** 2, case["C"]
        w, m = _rot_work(N, nl, Y * (kk - 1))
        w = nl * N * (2 * C + 2 * Y + Y * kk * C) + 4 * nl * (nl + 1) * N
        m += nl * (2 * (C + Y * kk) * _ntt_mults(N) + 2 * Y * kk * C * N)
    return {"bytes": 8 * w, "flops": 2 * m}


# ------------------------------------------------------------------ exact ---

def _mul(a, b, q):
    """a * b mod q for 0 <= a, b < q < 2^50: the quotient to within one in float64, the rest mod 2^64."""
    bf = b.double() if torch.is_tensor(b) else float(b)
    r = a * b - (a.double() * bf / q).floor().long() * q
    r = torch.where(r < 0, r + q, r)
    return torch.where(r >= q, r - q, r)


@functools.lru_cache(None)
def _roots(q, N):
    """psi^rev(k) and psi^-rev(k), psi the smallest primitive 2N-th root of unity mod q."""
    x = 2
    while pow(x, (q - 1) // 2, q) != q - 1:
        x += 1
    g = pow(x, (q - 1) // (2 * N), q)
    g2, psi, t = g * g % q, q, g
    for _ in range(N):
        psi, t = min(psi, t), t * g2 % q
    lg = N.bit_length() - 1
    rev = [int(format(k, "0%db" % lg)[::-1], 2) for k in range(N)]
    out = []
    for base in (psi, pow(psi, -1, q)):
        pw = [1] * N
        for j in range(1, N):
            pw[j] = pw[j - 1] * base % q
        out.append(torch.tensor([pw[r] for r in rev], dtype=torch.int64, device="cuda"))
    return out


def _ntt1(a, q, inverse):
    N = a.shape[-1]
    tw = _roots(q, N)[1 if inverse else 0]
    shape, a = a.shape, a.reshape(-1, N)
    m = N // 2 if inverse else 1
    while 1 <= m < N:
        v, w = a.view(a.shape[0], m, 2, N // (2 * m)), tw[m:2 * m].view(1, m, 1)
        x, y = v[:, :, 0], v[:, :, 1]
        if inverse:
            a = torch.stack(((x + y) % q, _mul((x - y) % q, w, q)), 2).view(-1, N)
            m //= 2
        else:
            y = _mul(y, w, q)
            a = torch.stack(((x + y) % q, (x - y) % q), 2).view(-1, N)
            m *= 2
    if inverse:
        a = _mul(a, pow(N, -1, q), q)
    return a.view(shape)


def _ntt(a, moduli, inverse=False):
    out = torch.empty_like(a)
    per = max(1, (1 << 25) // a.shape[-1])  # polynomials at a time
    for i, q in enumerate(moduli):
        src, dst = a[..., i, :].reshape(-1, a.shape[-1]), []
        for j in range(0, src.shape[0], per):
            dst.append(_ntt1(src[j:j + per], q, inverse))
        out[..., i, :] = torch.cat(dst).view(out[..., i, :].shape)
    return out


def _mulq(a, b, moduli):
    return torch.stack([_mul(a[..., i, :], b[..., i, :], q) for i, q in enumerate(moduli)], -2)


def _lift(v, moduli):
    return torch.stack([v % q for q in moduli], -2)


def _sum_mod(terms, moduli):
    acc = None
    for t in terms:
        acc = t if acc is None else acc + t
    return torch.stack([acc[..., i, :] % q for i, q in enumerate(moduli)], -2)


def _layer(ct, W, B, moduli):
    """out[m*B + b] = sum_g ct[g*B + b] * W[m, g], W [M][G][N] small integers."""
    M, G, N = W.shape
    x = _ntt(ct, moduli).view(G, B, 2, len(moduli), N)
    out = torch.empty((M, B) + tuple(x.shape[2:]), dtype=torch.int64, device="cuda")
    step = max(1, (1 << 23) // (max(G, 2 * B) * N))  # output channels at a time
    for m in range(0, M, step):
        w = _ntt(_lift(W[m:m + step], moduli), moduli)
        shape = (w.shape[0],) + tuple(x.shape[1:])
        out[m:m + step] = _sum_mod((_mulq(x[g].expand(shape), w[:, g, None, None].expand(shape), moduli) for g in range(G)), moduli)
    return _ntt(out.view((M * B,) + tuple(x.shape[2:])), moduli, True)


def _pack(K, p, N):
    M, C, k, _ = K.shape
    area = p["Hw"] * p["Ww"]
    off = (p["Cw"] - 1) * area + (k - 1) * p["Ww"] + k - 1
    W = np.zeros((M, p["G"], N), dtype=np.int64)
    for c in range(C):
        g, cc = divmod(c, p["Cw"])
        for l in range(k):
            for j in range(k):
                W[:, g, off - cc * area - l * p["Ww"] - j] = K[:, c, l, j]
    return torch.from_numpy(W).cuda()


def _delta(moduli):
    Q = math.prod(moduli)
    return [Q // T_PLAIN % q for q in moduli]


def _step_exact(case, v, p, q):
    """The share is added to c0, then the layer, then the mask leaves the output slots of c0."""
    N, k, pad = case["N"], case["k"], case["pad"]
    oh, ow = p["Hw"] - k + 1, p["Ww"] - k + 1
    Hp, Wp = case["H"] + 2 * pad, case["W"] + 2 * pad
    Bh = p["B"] // p["Bw"]
    x = torch.zeros((p["G"] * p["Cw"], max(Hp, Bh * oh + k), max(Wp, p["Bw"] * ow + k)), dtype=torch.int64, device="cuda")
    x[:case["C"], pad:pad + case["H"], pad:pad + case["W"]] = v["share"]
    ct, area = v["ct"].clone(), p["Cw"] * p["Hw"] * p["Ww"]
    for g in range(p["G"]):
        for b in range(p["B"]):
            i0, j0 = b // p["Bw"] * oh, b % p["Bw"] * ow
            pk = x[g * p["Cw"]:(g + 1) * p["Cw"], i0:i0 + p["Hw"], j0:j0 + p["Ww"]].reshape(-1)
            for i, (qi, d) in enumerate(zip(q, _delta(q))):
                c0 = ct[g * p["B"] + b, 0, i, :area]
                c0.copy_((c0 + _mul(pk, d, qi)) % qi)
    y = _layer(ct, _pack(v["K"], p, N), p["B"], q).view(case["M"], p["B"], 2, len(q), N)
    Ho, Wo = Hp - k + 1, Wp - k + 1
    off = (p["Cw"] - 1) * p["Hw"] * p["Ww"] + (k - 1) * p["Ww"] + k - 1
    pos = off + torch.arange(oh, device="cuda")[:, None] * p["Ww"] + torch.arange(ow, device="cuda")
    slots = torch.zeros((case["M"], p["B"], len(q), oh, ow), dtype=torch.int64, device="cuda")
    for b in range(p["B"]):
        i0, j0 = b // p["Bw"] * oh, b % p["Bw"] * ow
        h, w = min(oh, Ho - i0), min(ow, Wo - j0)
        for i, (qi, d) in enumerate(zip(q, _delta(q))):
            r = _mul(v["mask"][:, i0:i0 + h, j0:j0 + w], d, qi)
            slots[:, b, i, :h, :w] = (y[:, b, 0, i][:, pos[:h, :w]] - r) % qi
    return [y[:, :, 1].reshape(-1, len(q), N).contiguous(), slots.view(-1, len(q), oh * ow)]


def _galois(a, g, moduli):
    """X -> X^g on the last axis."""
    N = a.shape[-1]
    src = torch.arange(N, device="cuda") * pow(g, -1, 2 * N) % (2 * N)
    b = a[..., src % N]
    return torch.stack([torch.where(src < N, b[..., i, :], -b[..., i, :] % q) for i, q in enumerate(moduli)], -2)


def _rotate(ct, key_ntt, g, q, sp):
    """Key-switched rotation of ct [n][2][L][N]: one digit per limb, rounding division by sp."""
    qp, s = q + (sp,), _galois(ct, g, q)
    u = [torch.zeros_like(ct[:, 0, :1]).expand(-1, len(qp), -1).clone() for _ in range(2)]
    for j in range(len(q)):
        d = _ntt(_lift(s[:, 1, j], qp), qp)
        for c in range(2):
            u[c] = _sum_mod((u[c], _mulq(d, key_ntt[j, c].expand_as(d), qp)), qp)
    out = torch.empty_like(ct)
    for c in range(2):
        w = _ntt(u[c], qp, True)
        cen = torch.where(w[:, -1] > (sp - 1) // 2, w[:, -1] - sp, w[:, -1])
        for i, qi in enumerate(q):
            out[:, c, i] = _mul((w[:, i] - cen) % qi, pow(sp, -1, qi), qi)
    out[:, 0] = _sum_mod((out[:, 0], s[:, 0]), q)
    return out


def _zp_weights(case, K, q):
    """[kk][Y][C] plaintexts with constant slot rows, SIMD-encoded mod P and lifted centred into q."""
    N, P, Y = case["N"], _plain_prime(), (case["M"] + 1) // 2
    lg = N.bit_length() - 1
    idx = [[int(format((e - 1) // 2, "0%db" % lg)[::-1], 2) for e in es] for es in
           ([pow(5, c, 2 * N) for c in range(N // 2)], [2 * N - pow(5, c, 2 * N) for c in range(N // 2)])]
    Kp = torch.zeros((2 * Y,) + tuple(K.shape[1:]), dtype=torch.int64, device="cuda")
    Kp[:case["M"]] = K
    Kp = Kp.view(Y, 2, case["C"], -1).permute(3, 0, 2, 1)  # [kk][Y][C][row]
    for i in range(Kp.shape[0]):
        A = torch.zeros(Kp.shape[1:3] + (N,), dtype=torch.int64, device="cuda")
        for row in range(2):
            A[..., torch.tensor(idx[row], device="cuda")] = Kp[i, ..., row:row + 1].expand(-1, -1, N // 2)
        a = _ntt(A.unsqueeze(-2), (P,), True).squeeze(-2)
        yield _ntt(_lift(torch.where(a > (P - 1) // 2, a - P, a), q), q)


def exact(case, seed):
    kind, v = case["kind"], _inputs(case, seed)
    if kind == "products":
        return [_ntt(_mulq(_ntt(ct, q), pt.unsqueeze(1).expand_as(ct), q), q, True) for N, q, ct, pt in v["classes"]]
    q, N = _moduli(case), case["N"]
    if kind == "ctpt":
        x, n, o = _ntt(v["ct"], q), case["n"], case["n_out"]
        pr = _mulq(x, v["pt"].unsqueeze(1).expand_as(x), q)
        return _ntt(torch.stack([_sum_mod((pr[j] for j in range(s, n, o)), q) for s in range(o)]), q, True)
    if kind == "fc":
        Cw, No, G, Mp = _fc_part(case["C"], case["M"], N)
        W = np.zeros((Mp, G, N), dtype=np.int64)
        for m in range(case["M"]):
            for g in range(G):
                row = v["K"][m, g * Cw:(g + 1) * Cw]
                W[m // No, g, m % No * Cw + Cw - 1 - np.arange(row.size)] = row
        return _layer(v["ct"], torch.from_numpy(W).cuda(), 1, q)
    if kind in ("conv", "step", "host"):
        p = _part(case["C"], case["H"], case["W"], case["M"], case["k"], case["pad"], N)
        if kind == "step":
            return _step_exact(case, v, p, q)
        out = _layer(v["ct"], _pack(v["K"], p, N), p["B"], q)
        return out.cpu() if kind == "host" else out
    if kind == "net":
        return [_layer(ct, _pack(K, p, N), p["B"], q) for s, p, K, ct in v["layers"]]
    sp = _special(q)
    keys = [_ntt(k, q + (sp,)) for k in v["key"]]
    x = _ntt(v["ct"], q)
    if kind == "macrot":
        acc = None
        for i in reversed(range(case["n"])):
            pr = _ntt(_mulq(x, v["w"][i].expand_as(x), q), q, True)
            acc = pr if acc is None else _sum_mod((_rotate(acc, keys[0], 5, q, sp), pr), q)
        return acc
    k, step = case["k"], case["W"] + 2 * case["pad"] - case["k"] + 1
    prods = []
    for w in _zp_weights(case, v["K"], q):  # [Y][C][L][N] of one kernel offset
        prods.append(_ntt(torch.stack([_sum_mod((_mulq(x[c], wy[c].expand_as(x[c]), q) for c in range(case["C"])), q)
                                       for wy in w]), q, True))
    acc = prods[-1]
    for i in reversed(range(k * k - 1)):
        row = (i + 1) % k == 0
        acc = _sum_mod((_rotate(acc, keys[row], pow(5, step, 2 * N) if row else 5, q, sp), prods[i]), q)
    return acc
