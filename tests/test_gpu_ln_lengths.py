"""LayerNorm + quantization at the row lengths where the thread group or the chunks per thread change, both input types, and with
more rows than one grid takes (the code sums of a row leave in the iteration after it)."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("D", [1024, 1032, 1280, 1536, 1544, 2048, 2056, 2560, 3072, 3080, 4096, 5120, 6144, 6152, 8192, 8200, 16384])
def test_ln_quant_row_lengths(D, bf16):
    rep = parity.check_ln_quant(37, D, 4, bf16, seed=D)
    assert rep["bad"] == 0, rep


@pytest.mark.parametrize("rows,D,bits,bf16,rms", [(3001, 2048, 4, True, False), (1500, 4096, 8, True, True), (2500, 1536, 6, False, False),
                                                  (1203, 8192, 4, False, False), (1300, 8192, 4, True, False)])
def test_ln_quant_many_rows(rows, D, bits, bf16, rms):
    rep = parity.check_ln_quant(rows, D, bits, bf16, seed=rows, rms=rms)
    assert rep["bad"] == 0, rep


@pytest.mark.parametrize("rows,D,bf16", [(700, 6152, True), (601, 7168, True), (450, 12296, True), (333, 16376, True), (400, 8200, False),
                                         (3001, 512, False), (2500, 1280, False), (4001, 200, False)])
def test_ln_quant_row_forms(rows, D, bf16):
    """Two rows per group where the row does not fill it, and the float forms under a register bound; odd numbers of rows, more than
    one grid takes at a time."""
    rep = parity.check_ln_quant(rows, D, 4, bf16, seed=rows + D)
    assert rep["bad"] == 0, rep


@pytest.mark.parametrize("D", [200, 4096])
def test_factors_off_the_16_byte_boundary(D):
    """gamma~ and beta~ are plain float arrays: the same codes and sums wherever they start."""
    import torch
    from paper_2402_05628_b200 import binding as B
    dev, g = "cuda:0", torch.Generator(device="cuda:0").manual_seed(D)
    x = torch.randn(301, D, device=dev, generator=g).to(torch.bfloat16)
    gamma, beta = torch.randn(D + 4, device=dev, generator=g), torch.randn(D + 4, device=dev, generator=g)
    got = []
    for shift_g, shift_b in ((0, 0), (1, 0), (0, 2), (3, 1)):
        gm, bt = torch.empty(D + 4, device=dev), torch.empty(D + 4, device=dev)
        gm, bt = gm[shift_g:shift_g + D].copy_(gamma[:D]), bt[shift_b:shift_b + D].copy_(beta[:D])
        codes, sums = torch.zeros(301, D, device=dev, dtype=torch.uint8), torch.zeros(301, device=dev, dtype=torch.int32)
        B.repq_ln_quant(x, gm, bt, 1e-6, 0.3, 8, 4 | B.REPQ_BYTE_CODES, codes, sums)
        torch.cuda.synchronize()
        got.append((codes, sums))
    assert all(torch.equal(c, got[0][0]) and torch.equal(s, got[0][1]) for c, s in got[1:])
