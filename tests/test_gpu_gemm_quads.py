"""Byte codes out of the plain epilogue, where a thread takes two columns of four rows: output groups that change inside a warp's 64 columns,
row tiles that end inside the eight rows of a quad's lanes, every tile width, code sums of ragged rows."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,groups,bits", [
    (300, 624, 512, 3, 4), (257, 1248, 768, 3, 6), (1029, 768, 256, 1, 8), (643, 1152, 384, 3, 4),
    (3000, 2304, 768, 3, 4), (2100, 1536, 4096, 1, 6), (5003, 528, 128, 1, 4),
])
def test_plain_byte_codes_match_oracle(M, N, K, groups, bits):
    b = 4 | parity.BYTE_CODES
    parity.check_qgemm(M, N, K, b, b, out_kind="codes", groups=groups, out_bits=bits | (parity.BYTE_CODES if bits < 8 else 0),
                       want_acc=False, want_out_sum=True, give_sums=True, seed=M + N)
