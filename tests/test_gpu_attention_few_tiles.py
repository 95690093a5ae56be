"""Fused attention at the number of query tiles up to which narrow heads take visits of 128 keys, and at the edges of those visits."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Bn,H,Lq,Lk,dh,bits,bp,causal,s_p", [
    (37, 4, 9, 70, 64, 4, 4, False, 1.0), (149, 1, 9, 70, 64, 4, 4, False, 1.0),          # 148 and 149 tiles
    (1, 2, 40, 64, 64, 4, 4, False, 1.0), (1, 2, 40, 65, 48, 4, 4, False, 1.0), (1, 3, 130, 128, 16, 4, 4, False, 1.0),
    (2, 2, 129, 129, 64, 4, 4, True, 1.0), (1, 2, 260, 257, 64, 6, 4, False, 1.0), (1, 2, 200, 255, 32, 6, 6, True, 1.0),
    (160, 1, 129, 129, 64, 4, 8, True, 1.0), (80, 2, 66, 100, 64, 4, 4, False, 0.7), (160, 1, 20, 130, 64, 6, 4, False, 1.0),
    (1, 2, 90, 190, 64, 4, 6, False, 0.7),
    (31, 1, 9, 129, 64, 4, 4, False, 1.0), (32, 1, 9, 129, 64, 4, 4, False, 1.0), (2, 1, 140, 191, 64, 6, 6, True, 1.0),   # 31, 32 tiles
    (2, 1, 140, 192, 64, 6, 6, True, 1.0),
])
def test_attention_with_few_tiles_matches_oracle(Bn, H, Lq, Lk, dh, bits, bp, causal, s_p):
    parity.check_attention(Bn, H, Lq, Lk, dh, bits, bp, causal, seed=Lq + Lk + dh, s_p=s_p)


@pytest.mark.parametrize("Bn,H,Lq,Lk,dh,bits,bp,causal,spread", [
    (5, 8, 640, 5000, 64, 4, 8, False, 1.0), (5, 8, 640, 5000, 64, 6, 6, False, 1.0), (5, 8, 640, 5000, 32, 4, 4, False, 3.0),
    (5, 8, 640, 3000, 64, 4, 8, True, 1.0), (7, 8, 333, 577, 64, 6, 6, False, 2.0), (40, 6, 130, 197, 64, 4, 4, False, 3.0),
    (30, 6, 60, 67, 48, 6, 8, True, 1.0), (30, 6, 129, 129, 64, 4, 8, False, 1.0),
    (9, 32, 60, 67, 48, 6, 8, True, 1.0), (6, 16, 129, 129, 64, 4, 8, False, 1.0),
])
def test_an_items_output_does_not_depend_on_the_number_of_items(Bn, H, Lq, Lk, dh, bits, bp, causal, spread):
    """Calls of more tiles than SMs and of fewer take different kernels: the same bits, down to the last bit of the Softmax sum.  (A
    sum in another order moves a code at a tie of its rounding about once in 1e7 scores for rows this flat; 1e8 scores are compared.)"""
    import math
    import torch
    from paper_2402_05628_b200 import binding as B
    dev, D = "cuda:0", H * dh
    g = torch.Generator(dev).manual_seed(Lk + dh)
    make = lambda rows: torch.randint(0, 1 << bits, (rows, D), device=dev, generator=g, dtype=torch.uint8)   # noqa: E731
    q, k, v = make(Bn * Lq), make(Bn * Lk), make(Bn * Lk)
    step = math.sqrt(spread / ((1 << 2 * bits) / 12.0))           # logits of that standard deviation

    def run(first, items):
        out = torch.zeros(items * Lq, D, device=dev)
        d = B.AttentionDesc()
        d.batch_outer, d.batch_inner, d.Lq, d.Lk, d.d_h, d.bits_qkv = items, H, Lq, Lk, dh, bits | B.REPQ_BYTE_CODES
        for name, t, L in (("q", q, Lq), ("k", k, Lk), ("v", v, Lk)):
            setattr(d, name + "_codes", t[first * L:].data_ptr())
            setattr(d, "ld%s_bytes" % name, D)
            setattr(d, name + "_stride_outer", L * D)
            setattr(d, name + "_stride_inner", dh)
            setattr(d, "z_" + name, 1 << bits - 1)
            setattr(d, "s_" + name, 0.05 if name == "v" else step)
        d.alpha, d.causal, d.bits_p, d.s_p = 1.0 / math.sqrt(dh), int(causal), bp, 1.0
        d.out, d.out_kind, d.ldo, d.o_stride_outer, d.o_stride_inner, d.out_row_sum = out.data_ptr(), B.REPQ_OUT_F32, D, Lq * D, dh, None
        B.repq_attention(d)
        torch.cuda.synchronize()
        assert B.repq_device_status() == 0
        return out

    whole = run(0, Bn)
    tiles = (Lq + 127) // 128 * H
    assert Bn * tiles > torch.cuda.get_device_properties(0).multi_processor_count >= tiles
    for i in range(Bn):
        assert torch.equal(run(i, 1), whole[i * Lq:(i + 1) * Lq]), i
