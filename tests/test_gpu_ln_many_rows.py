"""bf16 rows of 2048 and 4096 elements: calls of many rows give a warp a row of its own.  The same codes and sums, bit for bit, as the same
rows in calls of few, which share a row among warps; both sides of the number of rows where the kernels change, strides, all widths."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,dim,ldx,bits,rms", [
    (7993, 4096, 4096, 4, False), (7991, 4096, 4096, 4, False), (9001, 4096, 4104, 8, False), (8500, 4096, 4096, "4b", True),
    (14801, 2048, 2048, 4, False), (14799, 2048, 2048, 6, False), (18001, 2048, 2056, "4b", True), (20000, 2048, 2048, 8, False),
])
def test_codes_of_many_rows_are_those_of_few(rows, dim, ldx, bits, rms):
    import torch
    from paper_2402_05628_b200 import binding as B
    dev = "cuda:0"
    bits = 4 | B.REPQ_BYTE_CODES if bits == "4b" else bits
    g = torch.Generator(dev).manual_seed(rows)
    x = (torch.randn(rows, ldx, device=dev, generator=g) * torch.exp(torch.randn(ldx, device=dev, generator=g)) + 0.5).to(torch.bfloat16)[:, :dim]
    gamma, beta = 1.0 + 0.1 * torch.randn(dim, device=dev, generator=g), 0.1 * torch.randn(dim, device=dev, generator=g)
    scale, zero = np.float32(6.0 / ((1 << (bits & 15)) - 1)), (1 << (bits & 15)) // 2 - 1

    def run(step):
        codes = torch.zeros(rows, B.code_row_bytes(dim, bits), dtype=torch.uint8, device=dev)
        sums = torch.full((rows,), -1, dtype=torch.int32, device=dev)
        for r in range(0, rows, step):
            B.repq_ln_quant(x[r:r + step], gamma, beta, 1e-6, scale, zero, bits, codes[r:r + step], sums[r:r + step],
                            B.REPQ_NORM_RMS if rms else B.REPQ_NORM_LAYERNORM)
        torch.cuda.synchronize()
        assert B.repq_device_status() == 0
        return codes, sums

    (c0, s0), (c1, s1) = run(rows), run(2500)
    assert torch.equal(c0, c1) and torch.equal(s0, s1)


def test_factors_of_any_size_and_values_that_are_not_finite():
    """Products far beyond the codes' range clip at either end, in either kernel; a row with a NaN or an infinity leaves the others alone."""
    import torch
    from paper_2402_05628_b200 import binding as B
    dev, rows, dim = "cuda:0", 9000, 4096
    g = torch.Generator(dev).manual_seed(3)
    x = torch.randn(rows, dim, device=dev, generator=g).to(torch.bfloat16)
    gamma = torch.randn(dim, device=dev, generator=g) * 10.0 ** torch.randint(-3, 12, (dim,), device=dev, generator=g)
    beta = torch.zeros(dim, device=dev)
    want = torch.nn.functional.layer_norm(x.double(), (dim,), gamma.double(), None, 1e-6) / 0.5
    for r, bad in ((17, float("nan")), (4000, float("inf"))):
        x[r, 5] = bad
    got = []
    for step in (rows, 2500):
        codes = torch.zeros(rows, dim, dtype=torch.uint8, device=dev)
        for r in range(0, rows, step):
            B.repq_ln_quant(x[r:r + step], gamma, beta, 1e-6, np.float32(0.5), 7, 4 | B.REPQ_BYTE_CODES, codes[r:r + step], None)
        torch.cuda.synchronize()
        got.append(codes)
    assert torch.equal(got[0], got[1])
    keep = torch.ones(rows, dtype=torch.bool, device=dev)
    keep[[17, 4000]] = False
    clear = ((want - want.floor() - 0.5).abs() > 1e-4 * want.abs().clamp(min=1.0)) & keep[:, None]     # off a tie by more than float32 moves t
    assert bool((got[0].double() == (want.round() + 7).clamp(0, 15))[clear].all())
