"""Blocks with packed weights: all four matrices expanded by one kernel beside the first LayerNorm where the workspace has the room, one
by one or inside the GEMMs in smaller workspaces; the same bits, also where the weights are the work of the kernel just ahead."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _block(bits, batch):
    import torch
    from paper_2402_05628_b200.engine import QuantBlock
    from workloads import make_block_inputs
    w = make_block_inputs("c1_vit_s", batch=batch)
    w.cfg = dict(w.cfg, bits_a=bits, bits_w=bits, bits_p=bits)
    blk = QuantBlock(w, weight_storage="packed")
    return blk, torch.from_numpy(np.ascontiguousarray(w.x)).to(blk.device).to(blk.act_dtype)


@pytest.mark.parametrize("bits,batch", [(4, 1), (6, 1), (4, 8), (6, 9)])
def test_workspaces_of_every_size_give_the_same_bits(bits, batch):
    import torch
    from paper_2402_05628_b200 import binding as B
    blk, x = _block(bits, batch)
    d = blk.desc(batch)
    total, D, mlp = B.repq_block_workspace_bytes(d), blk.cfg["D"], blk.cfg["MLP"]
    sizes = [k * n for n, k in ((3 * D, D), (D, D), (mlp, D), (D, mlp))]
    got = {}
    # with room for all four; for the largest one alone; for none
    for name, nbytes in (("all", total), ("one", total - sum(sizes) + max(sizes)), ("none", total - sum(sizes))):
        ws = torch.full((nbytes // 256 * 256,), 0xEE, dtype=torch.uint8, device=x.device)
        y = torch.zeros(x.shape, dtype=blk.out_dtype, device=x.device)
        for _ in range(3):
            B.repq_block_forward(d, blk.params(), x, y, ws)
        torch.cuda.synchronize()
        got[name] = y
    assert B.repq_device_status() == 0
    assert torch.equal(got["all"], got["one"]) and torch.equal(got["all"], got["none"])


@pytest.mark.parametrize("bits,batch", [(4, 1), (6, 6)])
def test_packed_weights_of_a_block_written_just_ahead(bits, batch):
    """Every pass finds other weights, written by copies queued right before it; compared with the device idle in between."""
    import torch
    from paper_2402_05628_b200 import binding as B
    blk, x = _block(bits, batch)
    d, p = blk.desc(batch), blk.params()
    ws = torch.empty(B.repq_block_workspace_bytes(d), dtype=torch.uint8, device=x.device)
    linears = [blk.qkv, blk.proj, blk.fc1, blk.fc2]
    g = torch.Generator(x.device).manual_seed(bits)
    sets = [[torch.randint(0, 256, w.codes.shape, device=x.device, generator=g, dtype=torch.uint8) for w in linears] for _ in range(8)]
    got = []
    for idle in (True, False):
        outs = []
        for s in sets:
            for w, c in zip(linears, s):
                w.codes.copy_(c)
            if idle:
                torch.cuda.synchronize()
            y = torch.empty(x.shape, dtype=blk.out_dtype, device=x.device)
            B.repq_block_forward(d, p, x, y, ws)
            outs.append(y)
        torch.cuda.synchronize()
        got.append(outs)
    assert B.repq_device_status() == 0
    assert not torch.equal(got[0][0], got[0][1])
    assert all(torch.equal(a, b) for a, b in zip(*got))


@pytest.mark.parametrize("bits,batch", [(4, 1), (6, 6)])
def test_input_and_factors_of_a_block_written_just_ahead(bits, batch):
    """The first LayerNorm runs beside the expansion and has no wait of its own: its input and factors are the work of the kernels just
    ahead, other ones in every pass; compared with the device idle in between."""
    import torch
    from paper_2402_05628_b200 import binding as B
    blk, x = _block(bits, batch)
    d, p = blk.desc(batch), blk.params()
    ws = torch.empty(B.repq_block_workspace_bytes(d), dtype=torch.uint8, device=x.device)
    g = torch.Generator(x.device).manual_seed(bits)
    sets = [(torch.randn(x.shape, device=x.device, generator=g).to(x.dtype), 1.0 + torch.randn(blk.ln1_g.shape, device=x.device, generator=g),
             torch.randn(blk.ln1_b.shape, device=x.device, generator=g)) for _ in range(8)]
    got = []
    for idle in (True, False):
        outs = []
        for s in sets:
            for t, v in zip((x, blk.ln1_g, blk.ln1_b), s):
                t.copy_(v)
            if idle:
                torch.cuda.synchronize()
            y = torch.empty(x.shape, dtype=blk.out_dtype, device=x.device)
            B.repq_block_forward(d, p, x, y, ws)
            outs.append(y)
        torch.cuda.synchronize()
        got.append(outs)
    assert B.repq_device_status() == 0
    assert not torch.equal(got[0][0], got[0][1])
    assert all(torch.equal(a, b) for a, b in zip(*got))
