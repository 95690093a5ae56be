"""Common epilogue of the integer GEMM over many tiles per CTA (its column and row terms are prepared a tile ahead, in two buffers),
with ragged rows and columns, for each form that is fixed at compile time and for the one that follows the parameters.  At K = 128 a
bf16 residual comes in boxes; loads of it by row, and tiles by pairs of CTAs, are for K above 3072 (the last test)."""
import numpy as np
import pytest

from tests import parity

pytestmark = pytest.mark.gpu

FORMS = [dict(), dict(gelu=True), dict(residual="bf16"), dict(residual="f32"), dict(gelu=True, residual="bf16")]
# (bf16 outputs are compared to one of their own ulps, which the tail of GELU, accurate to 1e-7 |v|, does not keep: f32 and codes have it)
CASES = [(kw, out) for kw in FORMS for out in ("f32", "bf16", "codes") if not (kw.get("gelu") and out == "bf16")]


@pytest.mark.parametrize("kw,out_kind", CASES, ids=lambda v: v if isinstance(v, str) else "-".join("%s" % e for e in v.values()) or "plain")
def test_gemm_over_many_tiles_matches_oracle(kw, out_kind):
    b = 4 | parity.BYTE_CODES
    parity.check_qgemm(9001, 1104, 128, b, b, out_kind=out_kind, out_bits=b, want_acc=False, want_out_sum=out_kind == "codes",
                       give_sums=True, seed=len(out_kind) + len(kw), **kw)


def test_rotated_columns_over_many_tiles_match_oracle():
    parity.check_qgemm_pair_step(6006, 1152, 128, 4 | parity.BYTE_CODES, "rope", seed=3, L=77, dh=32)


@pytest.mark.parametrize("M,N,K,out_kind", [
    (14203, 1000, 3200, "bf16"),    # 444 tiles of 128 x 256, three rounds (224 by pairs would be four): residual loaded by row
    (12001, 1104, 3088, "bf16"),    # 235 tiles of 256 x 256 on 74 pairs of CTAs (four rounds; 470 single ones take longer)
    (12001, 1104, 3088, "codes"),   # the same by pairs, to codes
])
def test_gemm_of_long_k_over_many_tiles(M, N, K, out_kind):
    """Against float64 on the same device (integer sums below 2^53: exact).  Tolerances: half an ulp of bf16 for the output and 2^-22 of
    the addends for the float32 steps ahead of it; codes may differ where the quotient is that close to a rounding tie."""
    import torch
    from paper_2402_05628_b200 import binding as B
    dev, b = "cuda:0", 4 | parity.BYTE_CODES
    g = torch.Generator(dev).manual_seed(M + len(out_kind))
    a = torch.randint(0, 16, (M, K), device=dev, generator=g, dtype=torch.uint8)
    w = torch.randint(0, 16, (N, K), device=dev, generator=g, dtype=torch.uint8)
    s_w = 0.01 * (1.0 + torch.rand(N, device=dev, generator=g))
    z_w = torch.randint(0, 16, (N,), device=dev, generator=g, dtype=torch.int32)
    bias = torch.randn(N, device=dev, generator=g)
    s_a, z_a = float(np.float32(0.02)), 7
    value = s_a * s_w.double() * ((a.double() - z_a) @ (w.double() - z_w.double()[:, None]).T)
    addends = value.abs() + bias.double().abs()
    value += bias.double()
    kw = dict(s_w=s_w, z_w=z_w, bias=bias, a_row_sum=a.int().sum(1, dtype=torch.int32), w_row_sum=w.int().sum(1, dtype=torch.int32))
    if out_kind == "bf16":
        res = torch.randn(M, N, device=dev, generator=g).bfloat16()
        out = torch.zeros(M, N, dtype=torch.bfloat16, device=dev)
        d = B.gemm_desc(M, N, K, a, b, s_a, z_a, w, b, out, residual=res, out_kind=B.REPQ_OUT_BF16, **kw)
    else:
        s_o, z_o = float(np.float32(0.4)), 8
        out, sums = torch.zeros(M, N, dtype=torch.uint8, device=dev), torch.zeros(M, dtype=torch.int32, device=dev)
        d = B.gemm_desc(M, N, K, a, b, s_a, z_a, w, b, out, out_kind=B.REPQ_OUT_CODES, out_bits=b, out_scale=[s_o], out_zero=[z_o],
                        out_row_sum=sums, **kw)
    B.repq_qgemm(d, torch.empty(max(B.repq_qgemm_workspace_bytes(d), 16), dtype=torch.uint8, device=dev))
    torch.cuda.synchronize()
    assert B.repq_device_status() == 0
    if out_kind == "bf16":
        value += res.double()
        addends += res.double().abs()
        assert bool(((out.double() - value).abs() <= 2.0 ** -8 * value.abs() + 2.0 ** -22 * addends).all())
    else:
        t = value / s_o
        open_ = 2.0 ** -21 * addends / s_o
        low, high = (torch.clamp(torch.round(t + e) + z_o, 0, 15) for e in (-open_, open_))
        assert bool(((out >= low) & (out <= high)).all())
        assert bool(torch.equal(sums, out.int().sum(1, dtype=torch.int32)))


@pytest.mark.parametrize("M,N,K", [(12608, 384, 384), (9601, 768, 768), (9500, 560, 700), (19001, 192, 768)])
def test_residual_in_two_boxes_matches_oracle(M, N, K):
    """Short K and more tiles of 192 columns than SMs: the next tile's residual comes while this one's leaves; ragged rows and columns."""
    b = 4 | parity.BYTE_CODES
    parity.check_qgemm(M, N, K, b, b, out_kind="bf16", residual="bf16", want_acc=False, give_sums=True, seed=M)
