"""Softmax + log2 codes at the row lengths where the number of chunks per thread changes: the edges of five, six and eight chunks
of eight keys, with and without a causal mask, both score types."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("L", [256, 257, 320, 321, 384, 385, 512, 513, 577, 640, 641, 768, 769, 1024, 1025, 1280, 1281, 1536, 1537, 2048, 2049])
def test_softmax_codes_at_the_edges_of_chunks_per_thread(L, bf16, causal):
    bits = 8 if L % 3 == 0 else 6 if L % 3 == 1 else 4
    rep = parity.check_softmax_log2(L if causal else 67, L, bits, bf16, seed=L, causal_period=L if causal else 0, ld_pad=(L + 7) // 8 * 8)
    assert rep["bad"] == 0
