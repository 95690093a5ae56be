"""Workloads that stand for what users run through this framework: whole quantized blocks on device-resident batches and
on batches in host memory, the single stages that a program composes itself, and the calibration step.

A case is a dict of plain values.  `prepare` makes its inputs from the seed and its weights from the configuration alone
(a program loads its weights once and keeps them), `run` is one pass through the public entry points.  Sizes are those of
the block configurations and kernel sweeps of this repository, and of the ranges around them."""
import math
from collections import OrderedDict
from types import SimpleNamespace

import torch

from paper_2402_05628_b200 import binding as B
from paper_2402_05628_b200.engine import QuantBlock

DEV = "cuda:0"


# ------------------------------------------------------------------------------------------------ the cases

def vit(name, batch, seq, dim, mlp=0, bits=4, act="bf16", storage="bytes"):
    return dict(name=name, kind="block", form="vit", batch=batch, seq=seq, dim=dim, heads=dim // 64, mlp=mlp or 4 * dim,
                bits=bits, bits_p=bits, act=act, storage=storage, causal=False)


def decoder(name, batch, seq, form="llama", dim=4096, mlp=11008, storage="bytes"):
    return dict(name=name, kind="block", form=form, batch=batch, seq=seq, dim=dim, heads=dim // 128, mlp=mlp, bits=4, bits_p=8,
                act="bf16", storage=storage, causal=True)


def listed():
    return [
        # one image through a ViT-S block, float32 activations: the smallest call, latency and launches
        vit("block_vit_s_b1_f32", 1, 197, 384, act="f32"),
        # a serving batch of DeiT-B, W4A4
        vit("block_deit_b_b64", 64, 197, 768),
        # a smaller W6A6 batch with the weights kept packed (capacity option)
        vit("block_deit_b_b16_w6_packed", 16, 197, 768, bits=6, storage="packed"),
        # ViT-L at 384 x 384: long ragged rows
        vit("block_vit_l_b32", 32, 577, 1024),
        # LLaMA-7B-shaped layer in the paper's block form, prefill of 4 x 2048 tokens: the largest
        decoder("block_llama7b_4x2048", 4, 2048, form="paper"),
        # the LLaMA block form (mean-free norm, rotary embedding, gated MLP): one ordinary prompt of an odd length
        decoder("block_llama_1x777", 1, 777),
        # and a short prompt, where a layer is one pass over its weights
        decoder("block_llama_1x48", 1, 48),
        # DeiT-B over four batches in pinned host memory, copies in and out included
        dict(name="host_deit_b_4x64", kind="host", batches=4, batch=64, seq=197, dim=768, heads=12, mlp=3072, bits=4, bits_p=4,
             act="bf16", storage="bytes", causal=False, form="vit"),
        # stages on their own, as in the kernel sweeps: LayerNorm + quantization to packed codes
        dict(name="ln_quant_32768x4096", kind="ln", rows=32768, dim=4096, bits=4, byte_codes=False, act="bf16", rms=False),
        # Softmax + log2 codes of 8 images x 16 heads x 577 queries
        dict(name="softmax_log2_73856x577", kind="softmax", rows=73856, length=577, bits=4, act="f32", causal=False),
        # the integer GEMM, W8A8
        dict(name="qgemm_w8a8_16384x4096x4096", kind="gemm", M=16384, N=4096, K=4096, bits=8, packed=False, out="bf16"),
        # calibration: per-channel dual clipping of one DeiT-S LayerNorm (32 images)
        dict(name="dual_clip_6304x384", kind="clip", rows=6304, dim=384, bits=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["vit", "vit", "vit", "decoder", "decoder", "host", "ln", "softmax", "gemm", "gemm", "clip"])
    if kind in ("vit", "host"):
        dim = rng.choice([384, 768, 1024])
        bits = rng.choice([4, 4, 6])
        seq = _log(rng, 50, 577)
        batch = min(_log(rng, 1, 64), 18464 // seq)
        case = vit("", batch, seq, dim, bits=bits, act="f32" if rng.random() < 0.25 else "bf16",
                   storage="packed" if rng.random() < 0.25 else "bytes")
        if kind == "host":
            case.update(kind="host", batches=rng.randint(1, 5), batch=max(1, min(batch, 12608 // seq * 768 // dim)), act="bf16")
    elif kind == "decoder":
        seq = _log(rng, 16, 2048)
        big = rng.random() < 0.5
        case = decoder("", min(_log(rng, 1, 4), max(1, 4096 // seq)), seq, form=rng.choice(["llama", "llama", "paper"]),
                       dim=4096 if big else 2048, mlp=11008 if big else 5504, storage="packed" if rng.random() < 0.2 else "bytes")
    elif kind == "ln":
        dim = rng.choice([384, 768, 1024, 1536, 2048, 4096, 8192])
        case = dict(kind="ln", rows=_log(rng, 1000, (32768 * 4096) // dim), dim=dim, bits=rng.choice([4, 6, 8]),
                    byte_codes=rng.random() < 0.5, act="f32" if rng.random() < 0.2 else "bf16", rms=rng.random() < 0.3)
        if case["act"] == "f32":
            case["rows"] = max(1000, case["rows"] // 2)
    elif kind == "softmax":
        length = rng.choice([197, 577, 2048, 8192, _log(rng, 50, 4096)])
        causal = length >= 1024 and rng.random() < 0.5
        case = dict(kind="softmax", rows=_log(rng, 64, (73856 * 577) // length), length=length, bits=rng.choice([4, 4, 6, 8]),
                    act="bf16" if rng.random() < 0.2 else "f32", causal=causal)
    elif kind == "gemm":
        N, K = rng.choice([(2304, 768), (768, 768), (3072, 768), (768, 3072), (3072, 1024), (1024, 4096), (4096, 4096), (12288, 4096),
                           (11008, 4096), (4096, 11008)])
        most = min(65536, 16384 * 4096 * 4096 // (N * K))
        bits = rng.choice([4, 4, 8])
        case = dict(kind="gemm", M=_log(rng, min(2048, most // 2), most), N=N, K=K, bits=bits, packed=bits == 4 and rng.random() < 0.5,
                    out=rng.choice(["bf16", "residual", "codes", "gelu"]))
    else:
        dim = rng.choice([192, 384, 768, 1024, 2048, 4096])
        case = dict(kind="clip", rows=_log(rng, 500, 6304 * 384 // dim), dim=dim, bits=rng.choice([4, 4, 6, 8]))
    case.pop("name", None)
    return case


# ------------------------------------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, device=DEV, generator=g)


def _channels(g, dim, massive):
    """Per-channel magnitude (log-normal, a few outlier or massive channels) and mean shift of a LayerNorm input."""
    c = torch.exp(_randn(g, dim))
    if massive:
        c[torch.arange(4, device=DEV) * (dim // 4) + dim // 8] = 1000.0
    else:
        n_out = max(1, dim // 100)
        c[torch.randperm(dim, device=DEV, generator=g)[:n_out]] *= 50.0
    return c, _randn(g, dim) * 0.5 * c


def _norm(x, gamma, beta, eps, rms):
    f = torch.nn.functional
    return f.rms_norm(x, x.shape[-1:], gamma, eps) + beta if rms else f.layer_norm(x, x.shape[-1:], gamma, beta, eps)


def _bounds(t, dim=None):
    """0.1 / 99.9 percentiles, per tensor or per channel."""
    if dim is None:
        t = t.reshape(-1)
        t, dim = t[:: t.numel() // 2_000_000 + 1], 0
    t = torch.sort(t, dim=0).values
    n = t.shape[0]
    lo, hi = t[int(0.001 * (n - 1))], t[int(math.ceil(0.999 * (n - 1)))]
    return lo, torch.maximum(hi, lo + 1e-6)


def _rotate(t, base=10000.0):
    """Rotary embedding of [L, H, dh] on consecutive channel pairs."""
    L, _, dh = t.shape
    theta = base ** (-torch.arange(0, dh, 2, device=DEV, dtype=torch.float64) / dh)
    a = torch.arange(L, device=DEV, dtype=torch.float64)[:, None] * theta
    rot = torch.polar(torch.ones_like(a), a)[:, None, :]
    return torch.view_as_real(torch.view_as_complex(t.double().reshape(L, -1, dh // 2, 2)) * rot).reshape(t.shape).float()


_BLOCKS = OrderedDict()       # the last few blocks: weights are loaded once and kept, as a program keeps them


def _block(case):
    """QuantBlock of the case's configuration: random weights of that shape, clipping bounds from a full-precision pass over a
    calibration sequence, the query projection scaled so that Softmax rows are heavy-tailed (median top-1 probability 0.5)."""
    key = tuple(case[k] for k in ("form", "seq", "dim", "heads", "mlp", "bits", "bits_p", "act", "storage", "causal"))
    if key in _BLOCKS:
        _BLOCKS.move_to_end(key)
        return _BLOCKS[key]
    D, H, mlp, llama = case["dim"], case["heads"], case["mlp"], case["form"] == "llama"
    dh, eps, L = D // H, 1e-5 if case["causal"] else 1e-6, min(case["seq"], 256)
    g = _gen(7)
    c, shift = _channels(g, D, massive=case["causal"])
    affine = [1.0 + 0.1 * _randn(g, D), 0.1 * _randn(g, D), 1.0 + 0.1 * _randn(g, D), 0.1 * _randn(g, D)]
    n1 = 2 * mlp if llama else mlp
    W = {k: 0.02 * _randn(g, n, m) for k, n, m in (("qkv", 3 * D, D), ("proj", D, D), ("fc1", n1, D), ("fc2", D, mlp))}
    b = {k: 0.02 * _randn(g, w.shape[0]) for k, w in W.items()}
    if llama:
        for t in [affine[1], affine[3], *b.values()]:
            t.zero_()
    lin = lambda t, k: torch.nn.functional.linear(t, W[k], b[k])   # noqa: E731
    L = max(L, 64)
    x = _randn(g, L, D) * c + shift
    x1 = _norm(x, affine[0], affine[1], eps, llama)
    q, k, v = (t.reshape(L, H, dh) for t in lin(x1, "qkv").split(D, dim=1))
    if llama:
        q, k = _rotate(q), _rotate(k)
    s = torch.einsum("ihd,jhd->hij", q, k) / math.sqrt(dh)
    if case["causal"]:
        s = s.masked_fill(~torch.ones(L, L, dtype=torch.bool, device=DEV).tril(), float("-inf"))
    lo, hi = 0.0, 14.0
    for _ in range(16):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if float(torch.softmax(s * 2.0 ** mid, -1).amax(-1).median()) < 0.5 else (lo, mid)
    tau = 2.0 ** lo
    W["qkv"][:D] *= tau
    b["qkv"][:D] *= tau
    o = torch.einsum("hij,jhd->ihd", torch.softmax(s * tau, -1), v).reshape(L, D)
    x2 = _norm(lin(o, "proj") + x, affine[2], affine[3], eps, llama)
    h = lin(x2, "fc1")
    if llama:
        h = torch.nn.functional.silu(h[:, :mlp]) * h[:, mlp:]
    else:
        h = torch.nn.functional.gelu(h)
    np_ = lambda t: t.cpu().numpy()                                  # noqa: E731
    ln1, ln2 = _bounds(x1, 0), _bounds(x2, 0)
    w = SimpleNamespace(
        cfg=dict(B=case["batch"], L=case["seq"], D=D, H=H, MLP=mlp, bits_a=case["bits"], bits_w=case["bits"], bits_p=case["bits_p"],
                 act=case["act"], causal=case["causal"], eps=eps, arch="llama" if llama else "vit", rope_base=10000.0),
        ln1_gamma=np_(affine[0]), ln1_beta=np_(affine[1]), ln2_gamma=np_(affine[2]), ln2_beta=np_(affine[3]),
        ln1_lo=np_(ln1[0]), ln1_hi=np_(ln1[1]), ln2_lo=np_(ln2[0]), ln2_hi=np_(ln2[1]),
        w_qkv=np_(W["qkv"]), b_qkv=np_(b["qkv"]), w_proj=np_(W["proj"]), b_proj=np_(b["proj"]),
        w_fc1=np_(W["fc1"]), b_fc1=np_(b["fc1"]), w_fc2=np_(W["fc2"]), b_fc2=np_(b["fc2"]),
        bounds={n: tuple(float(e) for e in _bounds(t)) for n, t in (("q", q * tau), ("k", k), ("v", v), ("attn", o), ("hidden", h))},
        softmax_scale=1.0)
    while len(_BLOCKS) >= 3:
        _BLOCKS.popitem(last=False)
    _BLOCKS[key] = QuantBlock(w, device=DEV, weight_storage=case["storage"]), c, shift
    return _BLOCKS[key]


def _codes(g, rows, cols, bits, zero):
    """Bell-shaped codes around the zero point, as quantized activations and weights are; one per byte."""
    top = (1 << bits) - 1
    out = torch.empty(rows, cols, dtype=torch.uint8, device=DEV)
    for r in range(0, rows, 8192):
        t = _randn(g, min(8192, rows - r), cols)
        out[r:r + 8192] = t.mul_(top / 6.0).add_(zero).round_().clamp_(0, top)
    return out


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    act = torch.float32 if case.get("act") == "f32" else torch.bfloat16
    if kind in ("block", "host"):
        blk, c, shift = _block(case)
        rows = case["batch"] * case["seq"]
        make = lambda: (_randn(g, rows, case["dim"]) * c + shift).to(act)   # noqa: E731
        if kind == "block":
            x = make()
            return dict(kind=kind, blk=blk, x=x, y=torch.empty_like(x))
        xs = [make().cpu().pin_memory() for _ in range(case["batches"])]
        return dict(kind=kind, blk=blk, xs=xs, ys=[torch.empty_like(x).pin_memory() for x in xs])
    if kind == "ln":
        rows, D, bits = case["rows"], case["dim"], case["bits"] | (B.REPQ_BYTE_CODES if case["byte_codes"] else 0)
        c, shift = _channels(g, D, massive=D >= 2048)
        gamma, beta = 1.0 + 0.1 * _randn(g, D), 0.1 * _randn(g, D)
        lo, hi = _bounds(_norm(_randn(g, 2048, D) * c + shift, gamma, beta, 1e-6, case["rms"]), 0)
        s, z = B.repq_scale_zero_from_bounds(lo.cpu().numpy(), hi.cpu().numpy(), bits)
        g_t, b_t, s_t, z_t, _, _ = B.repq_fold_ln(gamma.cpu().numpy(), beta.cpu().numpy(), s, z, gamma[None].cpu().numpy(), None)
        x = torch.empty(rows, D, dtype=act, device=DEV)
        for r in range(0, rows, 16384):
            x[r:r + 16384] = _randn(g, min(16384, rows - r), D) * c + shift
        return dict(kind=kind, x=x, gamma=torch.from_numpy(g_t).to(DEV), beta=torch.from_numpy(b_t).to(DEV), s=s_t, z=z_t, bits=bits,
                    norm=B.REPQ_NORM_RMS if case["rms"] else B.REPQ_NORM_LAYERNORM,
                    codes=torch.zeros(rows, B.code_row_bytes(D, bits), dtype=torch.uint8, device=DEV),
                    row_sum=torch.zeros(rows, dtype=torch.int32, device=DEV))
    if kind == "softmax":
        # logits of power-law rows: one key of probability 0.3 .. 0.9, the others proportional to rank^-alpha
        rows, L = case["rows"], case["length"]
        ld = (L + 7) // 8 * 8 if act == torch.bfloat16 else (L + 3) // 4 * 4
        scores = torch.zeros(rows, ld, dtype=act, device=DEV)
        for r in range(0, rows, 8192):
            n = min(8192, rows - r)
            t = torch.rand(n, L, device=DEV, generator=g).mul_(L - 1).floor_().add_(1.0).log_()
            t *= -(1.0 + torch.rand(n, 1, device=DEV, generator=g))
            p1 = 0.3 + 0.6 * torch.rand(n, 1, device=DEV, generator=g)
            rest = torch.logsumexp(t, 1, keepdim=True)
            at = torch.randint(0, L, (n, 1), device=DEV, generator=g)
            t.scatter_(1, at, rest + torch.log(p1 / (1.0 - p1)))
            scores[r:r + n, :L] = t + 3.0 * _randn(g, n, 1)
        ldc = (L + 7) // 8 * (4 if case["bits"] == 4 else 8)
        return dict(kind=kind, scores=scores, L=L, bits=case["bits"], period=L if case["causal"] else 0,
                    codes=torch.zeros(rows, (ldc + 15) // 16 * 16, dtype=torch.uint8, device=DEV))
    if kind == "gemm":
        M, N, K, bits = case["M"], case["N"], case["K"], case["bits"]
        gw = _gen(11)
        top = (1 << bits) - 1
        za = top // 2 + 1
        a, w = _codes(g, M, K, bits, za), _codes(gw, N, K, bits, top / 2)
        asum, wsum = a.sum(1, dtype=torch.int32), w.sum(1, dtype=torch.int32)
        form = bits if case["packed"] or bits == 8 else bits | B.REPQ_BYTE_CODES
        if case["packed"]:
            a, w = a[:, 0::2] | (a[:, 1::2] << 4), w[:, 0::2] | (w[:, 1::2] << 4)
        s_w = 0.001 + 0.009 * torch.rand(N, device=DEV, generator=gw)
        z_w = torch.randint(top // 2 - 1, top // 2 + 3, (N,), device=DEV, generator=gw, dtype=torch.int32)
        bias = 0.02 * _randn(gw, N)
        kw, res = {}, None
        if case["out"] in ("codes", "gelu"):
            out = torch.zeros(M, N, dtype=torch.uint8, device=DEV)
            spread = 0.02 * 0.005 * (top / 6.0) ** 2 * math.sqrt(K)
            kw = dict(out_kind=B.REPQ_OUT_CODES, out_bits=bits | B.REPQ_BYTE_CODES, out_scale=(6.0 * spread / top,),
                      out_zero=(top // 2 if case["out"] == "codes" else 1,), gelu=case["out"] == "gelu")
        else:
            out = torch.zeros(M, N, dtype=torch.bfloat16, device=DEV)
            res = _randn(g, M, N).to(torch.bfloat16) if case["out"] == "residual" else None
            kw = dict(out_kind=B.REPQ_OUT_BF16, residual=res)
        d = B.gemm_desc(M, N, K, a, form, 0.02, za, w, form, out, s_w=s_w, z_w=z_w, a_row_sum=asum, w_row_sum=wsum, bias=bias, **kw)
        ws = torch.empty(max(B.repq_qgemm_workspace_bytes(d), 16), dtype=torch.uint8, device=DEV)
        return dict(kind=kind, desc=d, ws=ws, out=out, keep=(a, w, asum, wsum, s_w, z_w, bias, res))
    # clip: the normalised activations of a calibration batch
    rows, D = case["rows"], case["dim"]
    c, shift = _channels(g, D, massive=False)
    x = _norm(_randn(g, rows, D) * c + shift, 1.0 + 0.1 * _randn(g, D), 0.1 * _randn(g, D), 1e-6, False).contiguous()
    return dict(kind="clip", x=x, bits=case["bits"], lo=torch.zeros(D, device=DEV), hi=torch.zeros(D, device=DEV))


# ------------------------------------------------------------------------------------------------ one pass

def run(state):
    kind = state["kind"]
    if kind == "block":
        return state["blk"].forward(state["x"], state["y"])
    if kind == "host":
        state["blk"].forward_host(state["xs"], state["ys"])
        return state["ys"]
    if kind == "ln":
        B.repq_ln_quant(state["x"], state["gamma"], state["beta"], 1e-6, state["s"], state["z"], state["bits"], state["codes"],
                        state["row_sum"], state["norm"])
        return {"codes": state["codes"], "row_sum": state["row_sum"]}
    if kind == "softmax":
        B.repq_softmax_log2(state["scores"], state["L"], 1.0, state["bits"], state["codes"], causal_period=state["period"])
        return state["codes"]
    if kind == "gemm":
        B.repq_qgemm(state["desc"], state["ws"])
        return state["out"]
    B.repq_dual_clip(state["x"], state["bits"], state["lo"], state["hi"], None, iters=100, lr=0.01, alpha0=2.0)
    return {"lo": state["lo"], "hi": state["hi"]}


# ------------------------------------------------------------------------------------------------ what a pass needs

def work(case):
    kind = case["kind"]
    a = 4 if case.get("act") == "f32" else 2
    if kind in ("block", "host"):
        n = case.get("batches", 1) * case["batch"]
        D, L, mlp = case["dim"], case["seq"], case["mlp"]
        w = 4 * D * D + (3 if case["form"] == "llama" else 2) * D * mlp
        scores = n * case["heads"] * L * L * (0.5 if case["causal"] else 1.0)
        return {"bytes": 2 * n * L * D * a + w * (case["bits"] / 8 if case["storage"] == "packed" else 1),
                "flops": 2.0 * n * L * w + 4.0 * scores * (D // case["heads"])}
    if kind == "ln":
        code = 0.5 if case["bits"] == 4 and not case["byte_codes"] else 1
        return {"bytes": case["rows"] * (case["dim"] * (a + code) + 4), "flops": 8.0 * case["rows"] * case["dim"]}
    if kind == "softmax":
        n = case["rows"] * case["length"]
        return {"bytes": n * (a * (0.5 if case["causal"] else 1) + (0.5 if case["bits"] == 4 else 1)), "flops": 6.0 * n}
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        out = {"bf16": 2, "residual": 4, "codes": 1, "gelu": 1}[case["out"]]
        return {"bytes": (M * K + N * K) * (0.5 if case["packed"] else 1) + M * N * out, "flops": 2.0 * M * N * K}
    n = case["rows"] * case["dim"]
    return {"bytes": 4 * n + 8 * case["dim"], "flops": 12.0 * 100 * n}


def tolerance(case):
    kind = case["kind"]
    if kind in ("block", "host"):
        # inside, codes at a rounding tie may fall to either side; the output is the residual stream in bf16 (or float32)
        return {"rel": 5e-3, "max": 0.5}
    if kind == "ln":
        return {"rel": 0.0, "differ": 5e-3}        # ties of the rounding; one of them moves its row's sum
    if kind == "softmax":
        return {"rel": 0.0, "differ": 1e-3}
    if kind == "gemm":
        return {"rel": 4e-3, "differ": 1e-3}       # bf16 outputs; codes at ties
    return {"rel": 1e-5, "max": 1e-3}              # float32 bounds out of a float64 iteration
