"""What a block keeps between passes (descriptor, parameters, workspace), on CPU: nothing of it may outlive what it was made from."""
import pytest


@pytest.fixture(scope="module")
def block():
    from paper_2402_05628_b200.build import build_library
    build_library()
    from paper_2402_05628_b200.engine import QuantBlock
    from workloads import make_block_inputs
    return QuantBlock(make_block_inputs("c1_vit_s", batch=1), device="cpu")


def test_parameters_follow_their_storage(block):
    d, p, ws = block._prepared(1)
    assert all(a is b for a, b in zip(block._prepared(1), (d, p, ws)))          # nothing changed: the same objects
    old = block.qkv.codes.data
    try:
        block.qkv.codes.data = old.clone()                                       # another storage under the same tensor
        assert block._prepared(1)[1].qkv.w_codes == block.qkv.codes.data_ptr() != old.data_ptr()
    finally:
        block.qkv.codes.data = old
    g = block.ln1_g
    block.ln1_g = g.clone()
    assert block._prepared(1)[1].ln1_gamma_t == block.ln1_g.data_ptr() != g.data_ptr()
    block.ln1_g = g
    s, z = block.act_q["attn"]
    block.act_q["attn"] = (2 * s, z)
    assert block._prepared(1)[1].s_attn == pytest.approx(2 * s)
    block.act_q["attn"] = (s, z)
    assert block._prepared(1)[1].s_attn == pytest.approx(s)


def test_a_pass_gets_what_it_asked_for(block):
    """Another thread's pass over another batch size, at the moment where this one's is kept (played by a hook on the
    assignment): this one still returns its own descriptor and a workspace of its own size."""
    from paper_2402_05628_b200 import binding as B
    from paper_2402_05628_b200.engine import QuantBlock
    need = {n: B.repq_block_workspace_bytes(block.desc(n)) for n in (1, 2)}

    class Interrupted(QuantBlock):
        inside = False

        def __setattr__(self, name, value):
            super().__setattr__(name, value)
            if name.startswith("_") and not Interrupted.inside:
                Interrupted.inside = True
                self._prepared(1)
                Interrupted.inside = False

    block.__class__ = Interrupted
    try:
        d, _, ws = block._prepared(2)
    finally:
        block.__class__ = QuantBlock
    assert d.batch == 2 and ws.numel() >= need[2] > need[1]
