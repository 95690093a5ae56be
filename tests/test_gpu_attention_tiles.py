"""Fused attention where a CTA walks several query tiles, at the edges of tiles and visits, and with a log-sqrt2 scale below 1
(4-bit codes then keep the table of operand pairs)."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Bn,H,Lq,Lk,dh,bits,bp,causal,s_p", [
    (24, 16, 129, 129, 64, 4, 4, False, 1.0),         # more tiles than CTAs, second tile of one row
    (20, 16, 130, 65, 32, 6, 6, False, 1.0),
    (12, 14, 150, 150, 128, 4, 8, True, 1.0),
    (10, 16, 200, 200, 96, 6, 4, True, 1.0),
    (1, 1, 1, 1, 64, 4, 4, False, 1.0), (1, 2, 128, 64, 64, 4, 4, False, 1.0), (2, 1, 33, 95, 16, 4, 4, True, 1.0),
    (2, 2, 140, 100, 64, 4, 4, False, 0.7), (1, 2, 70, 200, 64, 4, 8, False, 1.0),
])
def test_attention_tiles_match_oracle(Bn, H, Lq, Lk, dh, bits, bp, causal, s_p):
    parity.check_attention(Bn, H, Lq, Lk, dh, bits, bp, causal, seed=Lq + dh, s_p=s_p)
