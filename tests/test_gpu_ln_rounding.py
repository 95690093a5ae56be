"""LayerNorm + quantization, element by element where the general tests look away: values that are not numbers, and exact ties."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# every kind of group (some lanes, a warp, several warps, a block), full and ragged, and calls that give a warp a row of its own
FORMS = [(64, 70), (384, 70), (768, 70), (1536, 300), (2048, 70), (2048, 14900), (3072, 33), (4096, 70), (4096, 8100), (6152, 33), (16384, 17)]


def _codes(x, gamma, beta, zero, bits, rms=False):
    import torch
    from paper_2402_05628_b200 import binding as B
    codes = torch.zeros(x.shape[0], B.code_row_bytes(x.shape[1], bits), dtype=torch.uint8, device=x.device)
    B.repq_ln_quant(x, gamma, beta, 1e-6, np.float32(1.0), zero, bits, codes, None, B.REPQ_NORM_RMS if rms else B.REPQ_NORM_LAYERNORM)
    torch.cuda.synchronize()
    assert B.repq_device_status() == 0
    codes = codes[:, :x.shape[1] // 2 if bits == 4 else x.shape[1]]
    return torch.stack([codes & 15, codes >> 4], dim=2).flatten(1) if bits == 4 else codes


@pytest.mark.parametrize("bits", [4, 6])
@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("D,rows", FORMS)
def test_codes_of_rows_that_are_not_numbers(D, rows, bf16, bits):
    """A row with a NaN or an infinity has no mean: all of its codes are the highest one, or the lowest where some factor is so large
    that t might reach 2^22; the same at every row length."""
    import torch
    dev = "cuda:0"
    x = torch.randn(rows, D, device=dev, generator=torch.Generator(dev).manual_seed(D)).to(torch.bfloat16 if bf16 else torch.float32)
    for row, bad in ((3, float("nan")), (7, float("inf")), (9, float("-inf"))):
        x[row, D // 3] = bad
    beta = torch.zeros(D, device=dev)
    for gamma, code in ((3.0, (1 << bits) - 1), (1.0e9, 0)):
        got = _codes(x, torch.full((D,), gamma, device=dev), beta, 6, bits)[[3, 7, 9]]
        assert bool((got == code).all()), (gamma, got[:, :8])


@pytest.mark.parametrize("bits", [4, 6, 8])
@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("D,rows", FORMS)
def test_ties_round_to_even_before_the_zero_point_is_added(D, rows, bf16, bits):
    """t = k + 1/2 exactly (gamma~ = 0, so that t = beta~): Eq. 4 rounds t to the even neighbour and adds z afterwards, odd or even."""
    import torch
    dev, top = "cuda:0", (1 << bits) - 1
    x = torch.randn(rows, D, device=dev, generator=torch.Generator(dev).manual_seed(D)).to(torch.bfloat16 if bf16 else torch.float32)
    gamma, k = torch.zeros(D, device=dev), torch.arange(D, device=dev) % (2 * top + 7)
    for zero in (0, 6, 7, -3, 101):
        beta = k.float() - zero - 2.5
        want = (torch.round(beta.double()) + zero).clamp(0, top).to(torch.uint8)
        got = _codes(x, gamma, beta, zero, bits, rms=zero == 6)
        assert bool((got == want).all()), (zero, (got != want).nonzero()[:4])
