"""Float rows that a block asks for two iterations ahead (calls of many rows): every row has the codes it has in a call of few rows,
which asks for nothing ahead."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# (a block of 256 threads takes 64 rows of up to 128 elements at a time, 32 of 256: more than three turns of 148 SMs with at most eight
# blocks each are 227328 rows)
@pytest.mark.parametrize("rows,dim,ldx", [
    (227401, 64, 64), (227401, 128, 128), (227401, 256, 256),
    (40009, 384, 384), (40009, 384, 400), (40009, 768, 768), (40009, 1536, 1536),
])
def test_layernorm_of_many_rows_is_that_of_few(rows, dim, ldx):
    import torch
    from paper_2402_05628_b200 import binding as B
    dev = "cuda:0"
    g = torch.Generator(dev).manual_seed(dim)
    x = torch.randn(rows, ldx, device=dev, generator=g)[:, :dim]
    gamma, beta = 1.0 + 0.1 * torch.randn(dim, device=dev, generator=g), 0.1 * torch.randn(dim, device=dev, generator=g)

    def run(step):
        codes = torch.zeros(rows, B.code_row_bytes(dim, 4), dtype=torch.uint8, device=dev)
        sums = torch.zeros(rows, dtype=torch.int32, device=dev)
        for r in range(0, rows, step):
            B.repq_ln_quant(x[r:r + step], gamma, beta, 1e-6, np.float32(0.4), 7, 4, codes[r:r + step], sums[r:r + step], B.REPQ_NORM_LAYERNORM)
        return codes, sums

    (c0, s0), (c1, s1) = run(rows), run(500)
    assert torch.equal(c0, c1) and torch.equal(s0, s1)
