"""Batches in host memory: calls of several threads at once, and sequences of any length against the block on the device."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _block(batch, seed, **overrides):
    import torch
    from paper_2402_05628_b200.engine import QuantBlock
    from workloads import make_block_inputs
    blk = QuantBlock(make_block_inputs("c1_vit_s", batch=2, **overrides))
    rows, D = batch * blk.cfg["L"], blk.cfg["D"]
    rng = np.random.default_rng(seed)
    xs = [torch.from_numpy(rng.standard_normal((rows, D), dtype=np.float32)).to(blk.act_dtype).pin_memory() for _ in range(3)]
    expect = [blk.forward(x.to(blk.device)).cpu() for x in xs]
    return blk, xs, expect


def test_calls_of_two_threads_do_not_take_each_others_events():
    """Each thread has a block, a stream and buffers of its own; only the helper streams and events are the library's."""
    import torch
    work = [_block(batch, seed) for batch, seed in ((24, 1), (40, 2))]
    wrong = []

    def loop(blk, xs, expect):
        try:
            stream = torch.cuda.Stream()
            for i in range(25):
                n = 1 + i % 7
                ys = [torch.empty(x.shape, dtype=blk.out_dtype).pin_memory() for x in (xs * 3)[:n]]
                with torch.cuda.stream(stream):
                    blk.forward_host((xs * 3)[:n], ys)
                stream.synchronize()
                if not all(torch.equal(y, e) for y, e in zip(ys, (expect * 3)[:n])):
                    wrong.append(i)
        except Exception as e:                                  # noqa: BLE001  (reported by the main thread)
            wrong.append(e)

    threads = [threading.Thread(target=loop, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


@pytest.mark.parametrize("batch", [1, 5, 24, 65])               # (whole batches, two to eight pieces, ragged ones)
def test_sequences_of_any_length(batch):
    import torch
    from paper_2402_05628_b200 import binding as B
    blk, xs, expect = _block(batch, batch)
    blk.forward(xs[0].to(blk.device))
    torch.cuda.synchronize()
    before = B.repq_launch_count()
    blk.forward(xs[0].to(blk.device))
    per_block = B.repq_launch_count() - before
    bytes_in, per_batch = xs[0].numel() * xs[0].element_size(), {}
    for n in (1, 2, 4, 5, 9, 40):
        ys = [torch.zeros(x.shape, dtype=blk.out_dtype).pin_memory() for x in (xs * 14)[:n]]
        before = B.repq_launch_count()
        blk.forward_host((xs * 14)[:n], ys)
        torch.cuda.synchronize()
        per_batch[n] = (B.repq_launch_count() - before) / n / per_block
        assert all(torch.equal(y, e) for y, e in zip(ys, (expect * 14)[:n]))
    # pieces by the bytes they save against the gaps they add, at four batches as at five
    gap = 585 << 10
    most = min(8, bytes_in // (2685 << 10), xs[0].shape[0] // 2048, batch)
    for n, pieces in per_batch.items():
        assert pieces == (most if most > 1 and n * most * gap <= bytes_in else 1)


def test_pieces_of_wider_codes_are_parts_of_the_whole():
    """6-bit codes, and Softmax codes of 8 bits, which show a last bit of a Softmax sum soonest: pieces of 12 images have 144 attention
    tiles, the whole batch of 24 has 288, on either side of the number of SMs."""
    import torch
    for bits in (dict(bits_a=6, bits_w=6, bits_p=6), dict(bits_p=8)):
        blk, xs, expect = _block(24, 11, **bits)
        for n in (1, 5):
            ys = [torch.zeros(x.shape, dtype=blk.out_dtype).pin_memory() for x in (xs * 2)[:n]]
            blk.forward_host((xs * 2)[:n], ys)
            torch.cuda.synchronize()
            assert all(torch.equal(y, e) for y, e in zip(ys, (expect * 2)[:n]))
