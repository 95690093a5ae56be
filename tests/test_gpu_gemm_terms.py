"""Common epilogue of the integer GEMM over many tiles per CTA (its column and row terms are prepared a tile ahead, in two buffers),
with ragged rows and columns, for each form that is fixed at compile time and for the one that follows the parameters."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu

FORMS = [dict(), dict(gelu=True), dict(residual="bf16"), dict(residual="f32"), dict(gelu=True, residual="bf16")]
# (bf16 outputs are compared to one of their own ulps, which the tail of GELU, accurate to 1e-7 |v|, does not keep: f32 and codes have it)
CASES = [(kw, out) for kw in FORMS for out in ("f32", "bf16", "codes") if not (kw.get("gelu") and out == "bf16")]


@pytest.mark.parametrize("kw,out_kind", CASES, ids=lambda v: v if isinstance(v, str) else "-".join("%s" % e for e in v.values()) or "plain")
def test_gemm_over_many_tiles_matches_oracle(kw, out_kind):
    b = 4 | parity.BYTE_CODES
    parity.check_qgemm(9001, 1104, 128, b, b, out_kind=out_kind, out_bits=b, want_acc=False, want_out_sum=out_kind == "codes",
                       give_sums=True, seed=len(out_kind) + len(kw), **kw)


def test_rotated_columns_over_many_tiles_match_oracle():
    parity.check_qgemm_pair_step(6006, 1152, 128, 4 | parity.BYTE_CODES, "rope", seed=3, L=77, dh=32)
