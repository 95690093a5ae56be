"""Parameters written by the kernel just ahead in the stream: the entry points are ordinary stream-ordered work, so a GEMM may
take its weights, and a LayerNorm its factors, from a kernel that is still running when it is queued.  Every pass writes other
parameters into the same buffers; its result is compared with the same calls with the device idle in between."""
import pytest

pytestmark = pytest.mark.gpu

PASSES = 12


def _terms(torch, a, w):
    N = w.shape[0]
    return dict(s_w=torch.full((N,), 0.01, device=a.device), z_w=torch.full((N,), 8, device=a.device, dtype=torch.int32),
                a_row_sum=a.sum(1, dtype=torch.int32), w_row_sum=w.sum(1, dtype=torch.int32))


def _codes_gemm(B, torch, x, w, out, bits, out_bits):
    """out[M, N] = codes of x w^T: a producer of codes (or of packed codes) that later calls take as their weights."""
    (M, K), N = x.shape, w.shape[0]
    kw = _terms(torch, x, w)
    d = B.gemm_desc(M, N, K, x, bits, 0.05, 7, w, bits, out, out_kind=B.REPQ_OUT_CODES, out_bits=out_bits,
                    out_scale=(0.05 * 0.01 * 21 * K ** 0.5 / 3,), out_zero=(8,), **kw)
    d.operands = (x, w, kw)                                    # (the descriptor holds addresses only)
    return d, torch.empty(max(B.repq_qgemm_workspace_bytes(d), 16), dtype=torch.uint8, device=x.device)


@pytest.mark.parametrize("tokens,packed", [(16, False), (48, True), (300, False), (300, True)])
def test_weights_written_just_ahead(tokens, packed):
    import torch
    from paper_2402_05628_b200 import binding as B
    dev, g = "cuda:0", torch.Generator(device="cuda:0").manual_seed(tokens)
    draw = lambda *s: torch.randint(0, 16, s, device=dev, generator=g, dtype=torch.uint8)
    N, K, inner, bits = 4096, 1024, 2048, 4 | B.REPQ_BYTE_CODES
    weights = torch.zeros(N, K // 2 if packed else K, device=dev, dtype=torch.uint8)
    w_bits = 4 if packed else bits
    a = draw(tokens, K)
    out = torch.empty(tokens, N, device=dev)
    kw = _terms(torch, a, weights)                             # (code sums of zero: the same correction on both sides)
    d = B.gemm_desc(tokens, N, K, a, bits, 0.05, 7, weights, w_bits, out, **kw)
    ws = torch.empty(max(B.repq_qgemm_workspace_bytes(d), 16), dtype=torch.uint8, device=dev)
    makers = [_codes_gemm(B, torch, draw(N, inner), draw(K, inner), weights, bits, w_bits) for _ in range(PASSES)]
    got = []
    for idle in (True, False):
        outs = []
        for make, make_ws in makers:
            B.repq_qgemm(make, make_ws)
            if idle:
                torch.cuda.synchronize()
            B.repq_qgemm(d, ws)
            outs.append(out.clone())
        torch.cuda.synchronize()
        got.append(outs)
    assert B.repq_device_status() == 0
    assert not torch.equal(got[0][0], got[0][1])               # (the passes do differ)
    assert all(torch.equal(x, y) for x, y in zip(*got))


@pytest.mark.parametrize("D", [768, 4096])
def test_factors_written_just_ahead(D):
    import torch
    from paper_2402_05628_b200 import binding as B
    dev, g = "cuda:0", torch.Generator(device="cuda:0").manual_seed(D)
    bits = 4 | B.REPQ_BYTE_CODES
    factors = torch.zeros(4096, D, device=dev)                 # float32 output of a GEMM; two of its last rows are the factors
    x = torch.randn(64, D, device=dev, generator=g).to(torch.bfloat16)
    codes = torch.empty(64, D, device=dev, dtype=torch.uint8)
    sums = torch.empty(64, device=dev, dtype=torch.int32)
    makers = []
    for _ in range(PASSES):
        a = torch.randint(0, 16, (4096, 1024), device=dev, generator=g, dtype=torch.uint8)
        w = torch.randint(0, 16, (D, 1024), device=dev, generator=g, dtype=torch.uint8)
        kw = _terms(torch, a, w)
        d = B.gemm_desc(4096, D, 1024, a, bits, 0.05, 7, w, bits, factors, **kw)
        d.operands = (a, w, kw)
        makers.append((d, torch.empty(max(B.repq_qgemm_workspace_bytes(d), 16), dtype=torch.uint8, device=dev)))
    got = []
    for idle in (True, False):
        outs = []
        for make, make_ws in makers:
            B.repq_qgemm(make, make_ws)
            if idle:
                torch.cuda.synchronize()
            B.repq_ln_quant(x, factors[-1], factors[-2], 1e-6, 0.3, 8, bits, codes, sums)
            outs.append((codes.clone(), sums.clone()))
        torch.cuda.synchronize()
        got.append(outs)
    assert B.repq_device_status() == 0
    assert not torch.equal(got[0][0][0], got[0][1][0])
    assert all(torch.equal(x[0], y[0]) and torch.equal(x[1], y[1]) for x, y in zip(*got))
