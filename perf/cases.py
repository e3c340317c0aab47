"""Performance cases of the MixFP4 W4A4 linear layer: what is measured.

Each case is one pass that a user's program makes through the public entry
points of ``paper_2605_31035_gb300.ops``.  The kinds:

* ``linear``   the serving path: ``linear(x, w_q)``, i.e. online quantization of
  the activations and the GEMM against weights quantized once;
* ``fewrows``  the decode-time linear on the native FP4 variant;
* ``native``   the prefill linear on the native FP4 variant (activations
  quantized and split per call, weights split once);
* ``rotated``  the linear with the random Hadamard rotation of the activations
  fused into their quantization (weights rotated and quantized once);
* ``train``    one layer's training step on master weights: forward, the input
  gradient (stochastically rounded output gradient, transposed 2D weights)
  and the weight gradient (both operands down their columns, rotated along
  the tokens or with the output gradient stochastically rounded);
* ``quantize`` one large tensor quantized (weights or a batch of activations);
* ``fake``     the quantize-dequantize of the candidate-set / block-size study.

``exact`` restates Algorithm 1 in plain torch (the fp32 steps whose roundings
define the codes, bit for bit) and evaluates everything after the codes in
64 bits.
"""
import math

import torch

from paper_2605_31035_gb300 import ops

DEV = "cuda:0"

# ---------------------------------------------------------------------- cases


def listed():
    return [
        # One token of one sequence through a square projection: the smallest call.
        dict(name="decode_1", kind="linear", M=1, N=4096, K=4096, mode=0, pad=0),
        # A small decode batch through a 70B-class MLP projection.
        dict(name="decode_16", kind="linear", M=16, N=28672, K=8192, mode=0, pad=0),
        # A fuller decode batch on the native FP4 variant (8B MLP gate).
        dict(name="decode_64_native", kind="fewrows", M=64, N=14336, K=4096, mode=0),
        # Prefill of 2048 tokens, 8B attention projection.
        dict(name="prefill_attn", kind="linear", M=2048, N=4096, K=4096, mode=0, pad=0),
        # Prefill of 4096 tokens, 8B MLP gate / up and down projections.
        dict(name="prefill_gate", kind="linear", M=4096, N=14336, K=4096, mode=0, pad=0),
        dict(name="prefill_down", kind="linear", M=4096, N=4096, K=14336, mode=0, pad=0),
        # A ragged batch: a packed prompt of odd length out of a wider buffer.
        dict(name="ragged", kind="linear", M=777, N=3000, K=2816, mode=0, pad=64),
        # The attention projection with both operands as native FP4 operands.
        dict(name="native_attn", kind="native", M=2048, N=4096, K=4096, mode=0),
        # The Hadamard-rotated layer.
        dict(name="rotated", kind="rotated", M=8192, N=8192, K=8192, mode=0),
        # A training step of an attention projection over 4096 tokens.
        dict(name="train_attn", kind="train", T=4096, I=4096, O=4096, wgrad="rht"),
        # Offline quantization of a large tensor.
        dict(name="quantize_large", kind="quantize", M=65536, K=4096, mode=0),
        # Candidate-set study on a batch of activations.
        dict(name="fake_three", kind="fake", M=16384, K=4096, cand=11, block=16, bf16=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(rng, lo, hi, step):
    return max(lo, min(hi, _log(rng, lo, hi) // step * step))


def draw(rng):
    kind = rng.choice(["linear", "linear", "linear", "decode", "decode", "fewrows", "native", "rotated", "train",
                       "quantize", "fake"])
    if kind in ("decode", "fewrows"):
        M, N, K = _log(rng, 1, 64), _log(rng, 512, 28672), _mult(rng, 1024, 14336, 256)
        if rng.random() < 0.7:
            N = max(512, N // 64 * 64)
        c = dict(kind="linear" if kind == "decode" else "fewrows", M=M, N=N, K=K, mode=rng.choice([0, 0, 0, 1, 3]))
        if kind == "decode":
            c["pad"] = 0
        return c
    if kind in ("linear", "native"):
        M, N, K = _log(rng, 65, 8192), _log(rng, 256, 14336), _mult(rng, 512, 14336, 256)
        while 2.0 * M * N * K > 8.0e11:
            M = max(65, M // 2)
        if rng.random() < 0.7:
            N = max(256, N // 64 * 64)
        c = dict(kind=kind, M=M, N=N, K=K, mode=rng.choice([0, 0, 0, 1, 3]))
        if kind == "linear":
            c["pad"] = rng.choice([0, 0, 64])
        return c
    if kind == "rotated":
        M, N, K = _log(rng, 1, 8192), _mult(rng, 1024, 8192, 64), _mult(rng, 1024, 8192, 256)
        return dict(kind=kind, M=M, N=N, K=K, mode=0)
    if kind == "train":
        return dict(kind=kind, T=_mult(rng, 512, 4096, 256), I=_mult(rng, 512, 4096, 256),
                    O=_mult(rng, 512, 4096, 256), wgrad=rng.choice(["rht", "sr"]))
    if kind == "quantize":
        return dict(kind=kind, M=_log(rng, 16, 32768), K=_mult(rng, 1024, 8192, 16), mode=rng.choice([0, 0, 0, 1, 3]))
    return dict(kind=kind, M=_log(rng, 64, 16384), K=_mult(rng, 1024, 4096, 64), cand=rng.choice([3, 5, 11, 15]),
                block=rng.choice([8, 16, 32, 64]), bf16=rng.random() < 0.5)


def work(case):
    k = case["kind"]
    if k in ("quantize", "fake"):
        n = case["M"] * case["K"]
        if k == "quantize":
            return {"bytes": n * 2 + n // 2 + n // 16 + 4, "flops": 0}
        return {"bytes": n * (2 + (2 if case["bf16"] else 4)) + n // case["block"] + 4, "flops": 0}
    if k == "train":
        T, I, O = case["T"], case["I"], case["O"]
        return {"bytes": 2 * (T * I + T * O + O * I) + 4 * (T * O + T * I + O * I), "flops": 6 * T * I * O}
    M, N, K = case["M"], case["N"], case["K"]
    # the native variant keeps two E2M1 operands and one scale byte per block
    wbytes = N * K + N * K // 16 if k == "native" else N * K // 2 + N * K // 16
    return {"bytes": 2 * M * K + wbytes + 4 * M * N, "flops": 2 * M * N * K}


# --------------------------------------------------------------------- inputs
# Activations and gradients: Student-t (3 degrees of freedom) times 0.5, one
# percent of the channels 50 times larger; weights: N(0, 0.02) with a
# lognormal(0, 0.5) factor per output row (the distributions of synth.py,
# drawn on the GPU).


def _gen(seed, which):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + which)
    return g


def _activations(rows, K, seed, which, outliers=True, pad=0, scale=0.5):
    g = _gen(seed, which)
    out = torch.zeros(rows, K + pad, dtype=torch.bfloat16, device=DEV)[:, :K]
    gain = torch.ones(K, device=DEV)
    if outliers:
        gain[torch.randperm(K, generator=g, device=DEV)[:K // 100]] = 50.0
    step = max(1, (1 << 26) // K)
    for r0 in range(0, rows, step):
        r1 = min(rows, r0 + step)
        z = torch.randn(r1 - r0, K, generator=g, device=DEV)
        d = torch.zeros(r1 - r0, K, device=DEV)
        for _ in range(3):
            d += torch.randn(r1 - r0, K, generator=g, device=DEV).square_()
        out[r0:r1] = z / torch.sqrt(d / 3.0) * scale * gain
    return out


def _weights(N, K, seed, which):
    g = _gen(seed, which)
    w = torch.randn(N, K, generator=g, device=DEV) * 0.02
    return (w * torch.exp(torch.randn(N, 1, generator=g, device=DEV) * 0.5)).to(torch.bfloat16)


def _signs(seed):
    return torch.randint(0, 256, (16,), generator=_gen(seed, 9), dtype=torch.uint8, device=DEV)


def _inputs(case, seed):
    k = case["kind"]
    if k in ("quantize", "fake"):
        return dict(x=_activations(case["M"], case["K"], seed, 1))
    if k == "train":
        return dict(x=_activations(case["T"], case["I"], seed, 1), w=_weights(case["O"], case["I"], seed, 2),
                    dy=_activations(case["T"], case["O"], seed, 3, outliers=False, scale=1e-3), signs=_signs(seed))
    t = dict(x=_activations(case["M"], case["K"], seed, 1, pad=case.get("pad", 0)),
             w=_weights(case["N"], case["K"], seed, 2))
    if k == "rotated":
        t["signs"] = _signs(seed)
    return t


def prepare(case, seed):
    t = _inputs(case, seed)
    k = case["kind"]
    st = dict(case=case, **t)
    if k in ("linear", "fewrows"):
        st["wq"] = ops.mixfp4_quantize(st.pop("w"), case["mode"])
    elif k == "native":
        st["wn"] = ops.mixfp4_split_native(ops.mixfp4_quantize(st.pop("w"), case["mode"]),
                                           keep_residual=case["mode"] == 0)
    elif k == "rotated":
        st["wq"] = ops.mixfp4_quantize_rht(st.pop("w"), t["signs"], case["mode"])
    elif k == "train":
        st["sr_seed"] = int(seed) + 77
    return st


def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "linear":
        return ops.linear(st["x"], st["wq"], case["mode"])
    if k == "fewrows":
        return ops.mixfp4_gemm_native_fewrows(ops.mixfp4_quantize(st["x"], case["mode"]), st["wq"])
    if k == "native":
        q = ops.mixfp4_quantize(st["x"], case["mode"])
        return ops.mixfp4_gemm_native(ops.mixfp4_split_native(q, keep_residual=case["mode"] == 0), st["wn"])
    if k == "rotated":
        return ops.mixfp4_gemm(ops.mixfp4_quantize_rht(st["x"], st["signs"], case["mode"]), st["wq"])
    if k == "quantize":
        q = ops.mixfp4_quantize(st["x"], case["mode"])
        return q.codes, q.scales, q.tensor_scale
    if k == "fake":
        return ops.mixfp4_fake_quantize(st["x"], case["cand"], case["block"],
                                        torch.bfloat16 if case["bf16"] else torch.float32)
    # train: the three GEMMs of a layer's step
    x, w, dy, sg, seed = st["x"], st["w"], st["dy"], st["signs"], st["sr_seed"]
    wq = ops.mixfp4_quantize_2d(w)
    y = ops.mixfp4_gemm(ops.mixfp4_quantize(x), wq)
    dx = ops.mixfp4_gemm(ops.mixfp4_quantize_sr(dy, seed), ops.mixfp4_transpose_2d(wq))
    if case["wgrad"] == "rht":
        dw = ops.mixfp4_gemm(ops.mixfp4_quantize_colwise_rht(dy, sg), ops.mixfp4_quantize_colwise_rht(x, sg))
    else:
        dw = ops.mixfp4_gemm(ops.mixfp4_quantize_sr(dy, seed, offset=1, colwise=True), ops.mixfp4_quantize_colwise(x))
    return y, dx, dw


# ---------------------------------------------------------------------- exact


def _t(v):
    return torch.tensor(v, dtype=torch.float32, device=DEV)


def _e4m3(b):
    return b.clamp(max=448.0).to(torch.float8_e4m3fn).to(torch.float32)


def _to_codebook(m, book):
    """Round to nearest in `book`, a tie to the even position, saturating."""
    i = torch.zeros_like(m, dtype=torch.int8)
    for j in range(1, len(book)):
        mid = (book[j - 1] + book[j]) / 2
        i += (m >= mid) if j % 2 == 0 else (m > mid)
    return i


_E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)
_E1M2 = (0.0, 1.0, 2.0, 3.0, 4.0, 5.0, 6.0, 7.0)
_E3M0 = (0.0, 0.25, 0.5, 1.0, 2.0, 4.0, 8.0, 16.0)
# candidate: (divisor of the block maximum, codebook)
_CANDS = ((6.0, _E2M1), (7.0, _E1M2), (4.0, _E2M1), (16.0, _E3M0))
_MODE_CANDS = {0: (0, 1), 1: (0,), 2: (1,), 3: (0, 2)}


def _fma_chain(d):
    """fp32 fma chain of d^2 along the last dimension, from zero."""
    s = torch.zeros(d.shape[:-1], dtype=torch.float32, device=d.device)
    for i in range(d.shape[-1]):
        s = (s.double() + d[..., i].double().square()).float()
    return s


def _tree(s):
    """Pairwise tree of the fp32 sums along the last dimension."""
    while s.shape[-1] > 1:
        s = s[..., 0::2] + s[..., 1::2]
    return s[..., 0]


def _scale32(x):
    return x.abs().max().float() / _t(2688.0)


def _algorithm1(x, s32, cands, block=16, tile=False, sr=None):
    """Algorithm 1 on fp32 [rows, K]: the 64-bit values v * s8 * s32 with sign
    and the chosen candidate of each block (the later one on a tie)."""
    rows, K = x.shape
    out = torch.empty(rows, K, dtype=torch.float64, device=DEV)
    choice = torch.empty(rows, K // block, dtype=torch.uint8, device=DEV)
    step = max(16, (1 << 24) // K // 16 * 16)
    for r0 in range(0, rows, step):
        r1 = min(rows, r0 + step)
        xs = x[r0:r1].float()
        n = r1 - r0
        if tile and n % 16:
            xs = torch.cat([xs, xs.new_zeros(16 - n % 16, K)])
        a = (xs.abs() / s32 if s32.item() > 0 else torch.zeros_like(xs)).reshape(-1, K // block, block)
        B = a.amax(-1)
        if tile:
            B = B.reshape(-1, 16, K // 16).amax(1, keepdim=True).expand(-1, 16, -1).reshape(-1, K // 16)
        best = None
        for c in cands:
            div, book = _CANDS[c]
            s8 = _e4m3(B / _t(div))
            m = torch.where(s8[..., None] > 0, a / s8[..., None], torch.zeros_like(a))
            q = _t(book)[_to_codebook(m, book).long()]
            d = q * s8[..., None] - a
            g = min(block, 16)
            dc = d.reshape(*d.shape[:-1], block // g, g)
            S = _tree(_fma_chain(dc[..., 0::2]) + _fma_chain(dc[..., 1::2]))
            if tile:
                S = _tree(S.reshape(-1, 16, K // 16).transpose(1, 2).contiguous())
                S = S[:, None, :].expand(-1, 16, -1).reshape(-1, K // 16)
            if best is None:
                best = [S, s8, q, m, torch.full_like(S, c, dtype=torch.uint8)]
            else:
                w = S <= best[0]
                best = [torch.where(w, S, best[0]), torch.where(w, s8, best[1]),
                        torch.where(w[..., None], q, best[2]), torch.where(w[..., None], m, best[3]),
                        torch.where(w, torch.full_like(best[4], c), best[4])]
        S, s8, q, m, ch = best
        if sr is not None:
            seed, offset = sr
            e0 = torch.arange(r0 * K // 4, r1 * K // 4, device=DEV)
            eps = _uniforms(e0, seed, offset).reshape(m.shape)
            q1 = _round_up_below(m, eps, _E2M1)
            q2 = _round_up_below(m, eps, _E1M2)
            q = torch.where((ch == 1)[..., None], q2, q1)
        v = q.double() * s8.double()[..., None] * s32.double()
        v = torch.where(torch.signbit(xs).reshape(v.shape), -v, v).reshape(-1, K)
        out[r0:r1] = v[:n]
        choice[r0:r1] = ch[:n]
    return out, choice


def _round_up_below(m, eps, book):
    """Stochastic rounding: the upper neighbour iff eps is below the position
    of m between its neighbours; saturating at the largest value."""
    b = _t(book)
    i = torch.bucketize(m, b, right=True) - 1
    i = i.clamp(0, len(book) - 2)
    frac = (m - b[i]) / (b[i + 1] - b[i])
    q = torch.where(eps < frac, b[i + 1], b[i])
    return torch.where(m >= book[-1], b[-1], q)


def _uniforms(ctr, seed, offset):
    """Philox4x32-10: four 24-bit uniforms per counter value."""
    mask = 0xFFFFFFFF

    def mulhilo(m, x):
        lo, hi = x & 0xFFFF, x >> 16
        p0, p1 = m * lo, m * hi          # below 2^48
        t = p1 + (p0 >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (p0 & 0xFFFF)

    c = [ctr & mask, ctr >> 32, torch.full_like(ctr, offset & mask), torch.full_like(ctr, offset >> 32)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        h0, l0 = mulhilo(0xD2511F53, c[0])
        h1, l1 = mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return torch.stack([(w >> 8).float() * 2.0 ** -24 for w in c], dim=-1)


def _rotate(x, signs):
    """The sign flips and the 128-point Walsh-Hadamard transform (strides 1 to
    64, fp32) of every 128-element chunk of a row."""
    rows, K = x.shape
    bits = (signs.long()[:, None] >> torch.arange(8, device=DEV)) & 1
    flip = 1.0 - 2.0 * bits.reshape(128).float()
    v = x.float().reshape(rows, K // 128, 128) * flip
    h = 1
    while h < 128:
        p = v.reshape(rows, K // 128, 128 // (2 * h), 2, h)
        v = torch.stack([p[..., 0, :] + p[..., 1, :], p[..., 0, :] - p[..., 1, :]], dim=3)
        h *= 2
    return v.reshape(rows, K) * _t(128.0 ** -0.5)


def _values(x, mode=0, **kw):
    return _algorithm1(x, _scale32(x), _MODE_CANDS[mode], **kw)[0]


def exact(case, seed):
    t = _inputs(case, seed)
    k = case["kind"]
    x = t["x"]
    if k == "quantize":
        return None, None, x.abs().max().double().reshape(1) / 2688.0
    if k == "fake":
        cands = [c for c in range(4) if case["cand"] >> c & 1]
        v, _ = _algorithm1(x, _scale32(x), cands, block=case["block"])
        return v, None, x.abs().max().double().reshape(1) / 2688.0
    if k == "train":
        w, dy, sg, s = t["w"], t["dy"], t["signs"], int(seed) + 77
        wv = _values(w, tile=True)
        y = _values(x) @ wv.T
        dx = _values(dy, sr=(s, 0)) @ wv
        xt, dyt = x.t().contiguous(), dy.t().contiguous()
        if case["wgrad"] == "rht":
            a, b = _values(_rotate(dyt, sg)), _values(_rotate(xt, sg))
        else:
            a, b = _values(dyt, sr=(s, 1)), _values(xt)
        return y, dx, a @ b.T
    w = t["w"]
    if k == "rotated":
        x, w = _rotate(x, t["signs"]), _rotate(w, t["signs"])
    return _values(x, case["mode"]) @ _values(w, case["mode"]).T
