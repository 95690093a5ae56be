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
])
def test_attention_with_few_tiles_matches_oracle(Bn, H, Lq, Lk, dh, bits, bp, causal, s_p):
    parity.check_attention(Bn, H, Lq, Lk, dh, bits, bp, causal, seed=Lq + Lk + dh, s_p=s_p)
