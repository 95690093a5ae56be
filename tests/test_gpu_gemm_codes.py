"""Byte codes out of the integer GEMM's common epilogue for each width of the output quantizer (the pack instruction clips at a
shift that depends on it); scale folded into the column terms or applied last, one and three column groups, whole and ragged
tiles, the gated product."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [4, 6, 8])
@pytest.mark.parametrize("M,N,K,kw", [
    (300, 768, 768, dict()),
    (129, 576, 384, dict(groups=3)),
    (333, 1024, 256, dict(gelu=True)),
    (260, 400, 512, dict(residual="bf16")),
])
def test_byte_codes_match_oracle(M, N, K, kw, bits):
    b = 4 | parity.BYTE_CODES
    parity.check_qgemm(M, N, K, b, b, out_kind="codes", out_bits=bits | (parity.BYTE_CODES if bits < 8 else 0), want_acc=False,
                       want_out_sum=True, give_sums=True, seed=M + bits, **kw)


@pytest.mark.parametrize("bits", [4, 6, 8])
def test_byte_codes_of_the_gated_product(bits):
    parity.check_qgemm_pair_step(300, 512, 384, bits | (parity.BYTE_CODES if bits < 8 else 0), "glu", seed=bits)
