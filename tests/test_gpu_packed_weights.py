"""Packed weights: expanded into the workspace (K off the 64-code step, off the byte, few and many tokens), and the same block
output from the built-in scratch, which has no room for that."""
import numpy as np
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits_w", [4, 6 | parity.PACKED6])
@pytest.mark.parametrize("M,N,K", [(3, 70, 65), (70, 130, 72), (200, 96, 1000), (300, 640, 204), (1, 64, 4096)])
def test_packed_weights_match_oracle(M, N, K, bits_w):
    parity.check_qgemm(M, N, K, 4 | parity.BYTE_CODES, bits_w, out_kind="f32", want_acc=False, give_sums=True, seed=M + K)


def test_packed_block_in_the_built_in_scratch():
    import torch
    from paper_2402_05628_b200 import binding as B
    from paper_2402_05628_b200.engine import QuantBlock
    from workloads import make_block_inputs
    w = make_block_inputs("c1_vit_s", batch=8)
    blk = QuantBlock(w, weight_storage="packed")
    d = blk.desc(8)
    assert B.repq_block_workspace_bytes(d) > B.REPQ_STATIC_WORKSPACE_BYTES       # with the byte form; without it fits
    x = torch.from_numpy(np.ascontiguousarray(w.x)).to(blk.device).to(blk.act_dtype)
    y = blk.forward(x)
    ys = torch.empty_like(y)
    B.repq_block_forward_static(d, blk.params(), x, ys)
    torch.cuda.synchronize()
    assert B.repq_device_status() == 0 and torch.equal(y, ys)
