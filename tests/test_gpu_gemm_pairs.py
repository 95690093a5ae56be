"""The integer GEMM by pairs of CTAs (256 x 256 tiles, chosen for long K): rows that end in the first or in the second CTA of a
pair, ragged columns and K, every output kind and epilogue step, against the oracle."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,kw", [
    (2049, 2064, 5520, dict(out_kind="codes", out_bits=4 | parity.BYTE_CODES, want_out_sum=True)),      # one row in the last pair
    (2300, 2056, 5504, dict(out_kind="bf16", residual="bf16")),                                         # 252 rows: second CTA cut
    (1930, 2100, 5600, dict(out_kind="f32", residual="f32", gelu=True)),
    (2000, 2304, 5504, dict(out_kind="codes", groups=3, out_bits=6 | parity.BYTE_CODES, want_out_sum=True)),
    (2048, 2048, 5504, dict(out_kind="codes", gelu=True, out_bits=4)),                                  # packed codes
])
def test_pair_tiles_match_oracle(M, N, K, kw):
    b = 4 | parity.BYTE_CODES
    parity.check_qgemm(M, N, K, b, b, give_sums=True, seed=M, **dict(dict(want_acc=False), **kw))


@pytest.mark.parametrize("mode,N", [("rope", 2304), ("glu", 2048)])
def test_pair_tiles_with_a_pair_step(mode, N):
    parity.check_qgemm_pair_step(2000, N, 5504, 4 | parity.BYTE_CODES, mode, seed=N)


@pytest.mark.parametrize("M,N,K,kw", [
    (2049, 2032, 5520, dict(out_kind="codes", out_bits=4 | parity.BYTE_CODES, want_out_sum=True)),      # one row in the last pair
    (2300, 2040, 5504, dict(out_kind="bf16", residual="bf16")),                                         # 252 rows: second CTA cut
])
def test_pair_tiles_in_one_round(M, N, K, kw):
    """72 tiles for 74 pairs, where 128-row tiles of any width take two rounds or as long a main loop each."""
    b = 4 | parity.BYTE_CODES
    parity.check_qgemm(M, N, K, b, b, give_sums=True, seed=M, **dict(dict(want_acc=False), **kw))
