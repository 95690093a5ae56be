"""Fused attention by output form: byte codes by 16-byte stores have kernels of their own, every other form (packed codes, floats) another;
numbers of heads and tiles that are no powers of two, and visits that end inside a thread's 32 columns."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu

BYTES = parity.BYTE_CODES


@pytest.mark.parametrize("out_kind,out_bits", [("codes", 4 | BYTES), ("codes", 8), ("codes", 4), ("bf16", 8)])
@pytest.mark.parametrize("Bn,H,Lq,Lk,dh,bits,bp,causal", [
    (31, 7, 131, 103, 64, 4, 4, False),        # more tiles than CTAs, 7 heads, the last visit ends 7 columns into a thread's
    (3, 5, 70, 37, 48, 4, 4, False), (1, 3, 200, 200, 128, 4, 8, True), (2, 3, 66, 129, 64, 6, 6, False),
])
def test_every_output_form_matches_oracle(Bn, H, Lq, Lk, dh, bits, bp, causal, out_kind, out_bits):
    parity.check_attention(Bn, H, Lq, Lk, dh, bits, bp, causal, out_kind=out_kind, out_bits=out_bits, seed=Lk + H)
