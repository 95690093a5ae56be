"""Dual clipping out of sorted values: channels whose values crowd in few buckets, repeat, lie on one side of zero or coincide, at
counts off the vector width and at the sorted form's largest; and what infinities and NaN do to a channel and to no other."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(X, bits, iters, alpha0=2.0):
    import torch
    from paper_2402_05628_b200 import binding as B
    D = X.shape[1]
    dev = torch.device("cuda:0")
    lo, hi = torch.zeros(D, device=dev), torch.zeros(D, device=dev)
    loss = torch.zeros(2 * D, dtype=torch.float64, device=dev)
    B.repq_dual_clip(torch.from_numpy(X).to(dev), bits, lo, hi, loss, iters=iters, lr=0.01, alpha0=alpha0)
    return lo.cpu().numpy(), hi.cpu().numpy(), loss.cpu().numpy()


def _channels(n, rng):
    base = rng.standard_normal((n, 11)).astype(np.float32)
    base[0, 1] = 3000.0                                      # one value far out: the others share a bucket
    base[:, 2] = np.round(base[:, 2] * 2.0) / 2.0            # few distinct values, many on rounding ties
    base[:, 3] = np.abs(base[:, 3]) + 0.1                    # all above zero
    base[:, 4] = -np.abs(base[:, 4]) * 100.0                 # all below
    base[:, 5] = 1.25                                        # constant
    base[:, 6] = 0.0
    base[:, 7] *= 1e-38                                      # down to denormal numbers
    base[:, 8] = np.exp(3.0 * base[:, 8])                    # long tail
    base[:, 9] *= 1e30
    return base


@pytest.mark.parametrize("n,bits", [(1, 4), (5, 4), (9, 4), (64, 4), (1031, 4), (4098, 4), (22528, 4), (22529, 4), (513, 6)])
def test_dual_clip_of_crowded_channels(n, bits):
    """Both sides are float64 with sums in another order (relative error below 2^-53 n Q^2): the tolerances of the other
    dual-clipping checks, 1e-6 of the range for the bounds, 1e-9 for the objective at the start."""
    from oracle import repq_oracle as orc
    X = _channels(n, np.random.default_rng(n))
    lo, hi, loss = _run(X, bits, iters=32, alpha0=6.0)
    ref = orc.dual_clip(X, bits, iters=32, lr=0.01, alpha0=6.0)
    span = X.max(axis=0).astype(np.float64) - X.min(axis=0)
    same = span == 0.0                                       # nothing to learn: contracted extremes, no objective
    keep = 1.0 / (1.0 + np.exp(-6.0))
    ref["x_low"] = np.where(same, keep * X.min(axis=0), ref["x_low"])
    ref["x_up"] = np.where(same, keep * X.max(axis=0), ref["x_up"])
    ref["loss0"], ref["loss"] = np.where(same, 0.0, ref["loss0"]), np.where(same, 0.0, ref["loss"])
    assert np.all(np.abs(lo - ref["x_low"]) <= 1e-6 * span + 1e-7 * np.abs(ref["x_low"]) + 1e-45)
    assert np.all(np.abs(hi - ref["x_up"]) <= 1e-6 * span + 1e-7 * np.abs(ref["x_up"]) + 1e-45)
    D = X.shape[1]
    floor = 1e-12 * n * span ** 2
    assert np.all(np.abs(loss[:D] - ref["loss0"]) <= 1e-9 * ref["loss0"] + floor)
    assert np.all(np.abs(loss[D:] - ref["loss"]) <= 1e-5 * ref["loss"] + floor)


@pytest.mark.parametrize("n", [40, 3000])
def test_dual_clip_of_channels_with_infinities(n):
    X = _channels(n, np.random.default_rng(n))
    clean = _run(X, 4, iters=32)
    bad = X.copy()
    bad[3, 0], bad[n - 1, 8], bad[7, 9] = np.inf, np.nan, -np.inf
    lo, hi, _ = _run(bad, 4, iters=32)
    for d in range(X.shape[1]):
        if d in (0, 8, 9):
            assert np.isnan(lo[d]) and np.isnan(hi[d])
        else:
            assert lo[d] == clean[0][d] and hi[d] == clean[1][d]
