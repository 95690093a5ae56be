"""The integer GEMM for few tokens: against the oracle, and bit for bit against the warp-MMA kernel, which a caller that
withholds the row sums gets for the same problem."""
import pytest

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,kw", [
    (1, 64, 64, dict(out_kind="f32")),                                        # one token, one k-block
    (16, 200, 4096, dict(out_kind="f32", want_acc=True)),                     # ragged channels, K split over a cluster of 8
    (17, 4096, 1152, dict(out_kind="bf16", residual="bf16")),                 # token tile just exceeded
    (33, 384, 1000, dict(out_kind="f32", residual="f32", gelu=True)),         # K off the k-block
    (63, 1536, 384, dict(out_kind="codes", gelu=True, out_bits=4 | parity.BYTE_CODES, want_out_sum=True)),
    (100, 2304, 768, dict(out_kind="codes", groups=3, out_bits=6 | parity.BYTE_CODES, want_out_sum=True)),
    (197, 384, 1536, dict(out_kind="f32", residual="f32")),                   # several token tiles, the last one ragged
    (394, 768, 3072, dict(out_kind="bf16", residual="bf16")),
])
def test_few_tokens_match_oracle(M, N, K, kw):
    kw = dict(dict(want_acc=False), **kw)
    parity.check_qgemm(M, N, K, 4 | parity.BYTE_CODES, 4 | parity.BYTE_CODES, give_sums=True, seed=M + N, **kw)


@pytest.mark.parametrize("M,N,K", [(1, 96, 128), (8, 384, 2048), (48, 12288, 512), (63, 4992, 4096), (40, 96, 400)])
@pytest.mark.parametrize("mode", ["rope", "glu", "packed", "codes8"])
def test_few_tokens_same_bits_as_the_warp_mma_kernel(M, N, K, mode):
    import torch
    from paper_2402_05628_b200 import binding as B
    dev = "cuda:0"
    g = torch.Generator(device=dev).manual_seed(M + K)
    bits = 8 if mode == "codes8" else 4
    a = torch.randint(0, 1 << bits, (M, K), device=dev, generator=g, dtype=torch.uint8)
    w = torch.randint(0, 1 << bits, (N, K), device=dev, generator=g, dtype=torch.uint8)
    sums = dict(a_row_sum=a.sum(1, dtype=torch.int32), w_row_sum=w.sum(1, dtype=torch.int32))
    terms = dict(s_w=torch.rand(N, device=dev, generator=g) * 0.01 + 0.001, bias=torch.randn(N, device=dev, generator=g),
                 z_w=torch.randint(5, 10, (N,), device=dev, generator=g, dtype=torch.int32))
    scale = 0.05 * 0.006 * (1 << bits) ** 2 / 12 * K ** 0.5 / 3
    groups = 3 if mode == "rope" else 1
    table = torch.from_numpy(B.repq_rope_table(50, 32)).to(dev)
    step = dict(rope=table, rope_period=50, rope_dim=32, rope_groups=2) if mode == "rope" else dict(glu=mode == "glu")
    got = []
    for kw in (sums, {}):
        out = torch.zeros(M, N // 2 if mode in ("glu", "packed") else N, device=dev, dtype=torch.uint8)
        rs = torch.zeros(M, device=dev, dtype=torch.int32)
        d = B.gemm_desc(M, N, K, a, bits | B.REPQ_BYTE_CODES, 0.05, 7, w, bits | B.REPQ_BYTE_CODES, out, out_kind=B.REPQ_OUT_CODES,
                        out_bits=4 if mode == "packed" else bits | B.REPQ_BYTE_CODES, out_scale=(scale,) * groups,
                        out_zero=(1 << (bits - 1),) * groups, out_row_sum=rs, **step, **terms, **kw)
        B.repq_qgemm(d, torch.empty(max(B.repq_qgemm_workspace_bytes(d), 16), dtype=torch.uint8, device=dev))
        torch.cuda.synchronize()
        got.append((out, rs))
    assert B.repq_device_status() == 0
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


@pytest.mark.parametrize("limit", [1, 100_000])
def test_copies_asked_for_early_are_drained_when_a_wait_runs_out(limit):
    """A stage whose weights were asked for ahead and whose activations never are: the copy is waited for all the same before
    the kernel returns (code 77, the wait that ran out; 78 would be a copy that did not end), also where it is still in flight."""
    from paper_2402_05628_b200 import binding as B
    B.repq_bounded_wait_selftest(limit)
    assert B.repq_device_status(reset=True) == 77
    parity.check_qgemm(16, 384, 384, 4 | parity.BYTE_CODES, 4 | parity.BYTE_CODES, out_kind="f32", want_acc=False, give_sums=True)
    assert B.repq_device_status() == 0


@pytest.mark.parametrize("M,N,K,kw", [
    (48, 4096, 4096, dict(out_kind="bf16", residual="bf16")),                 # 48 tokens a tile, clusters of four
    (197, 768, 3072, dict(out_kind="bf16", residual="bf16")),                 # 32 tokens, clusters of four, the last tile ragged
    (80, 768, 3072, dict(out_kind="f32", residual="f32")),                    # 16 tokens, clusters of eight
    (394, 1024, 4096, dict(out_kind="bf16", residual="bf16")),                # the most CTAs clusters of two or four get
    (512, 1152, 384, dict(out_kind="codes", out_bits=4 | parity.BYTE_CODES, groups=3)),
    (777, 2048, 1408, dict(out_kind="bf16", residual="bf16")),                # many token tiles, or the 128-row kernel
])
def test_few_token_plans_match_oracle(M, N, K, kw):
    """Tokens per tile and K splits across the range in which the plan of the few-token kernel moves."""
    b = 4 | parity.BYTE_CODES
    parity.check_qgemm(M, N, K, b, b, give_sums=True, seed=M + N + K, want_acc=False, **kw)
