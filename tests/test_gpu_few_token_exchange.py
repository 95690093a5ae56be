"""Few-token GEMM: partial sums sent behind the ring (one CTA per SM, two per SM) and over it (token tiles of 96 and 128 in clusters),
shares that leave a CTA of the cluster without tokens, and ragged last tiles; the accumulators bit for bit."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,kw", [
    (48, 4096, 1152, dict(out_kind="bf16", residual="bf16")),                 # 200 KB a CTA
    (17, 4096, 768, dict(out_kind="f32", residual="f32")),
    (8, 384, 8192, dict(out_kind="f32")),                                     # eight CTAs, two chunks, one of them outside the matrix
    (16, 2048, 8192, dict(out_kind="bf16")),                                  # fewer CTAs than SMs that do not all fit one per SM
    (242, 1152, 11008, dict(out_kind="f32")), (483, 1024, 8192, dict(out_kind="bf16", residual="bf16")),      # over the ring
    (300, 768, 3072, dict(out_kind="codes", out_bits=4 | parity.BYTE_CODES, gelu=True, want_out_sum=True)),
])
def test_partial_sums_match_oracle(M, N, K, kw):
    b = 4 | parity.BYTE_CODES
    parity.check_qgemm(M, N, K, b, b, give_sums=True, seed=M + K, want_acc=True, **kw)
