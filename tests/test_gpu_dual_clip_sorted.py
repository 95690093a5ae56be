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


def _check_against_oracle(X, lo, hi, loss, bits):
    """Both sides are float64 with sums in another order (relative error below 2^-53 n Q^2): the tolerances of the other
    dual-clipping checks, 1e-6 of the range for the bounds, 1e-9 for the objective at the start."""
    from oracle import repq_oracle as orc
    n, D = X.shape
    ref = orc.dual_clip(X, bits, iters=32, lr=0.01, alpha0=6.0)
    span = X.max(axis=0).astype(np.float64) - X.min(axis=0)
    same = span == 0.0                                       # nothing to learn: contracted extremes, no objective
    keep = 1.0 / (1.0 + np.exp(-6.0))
    ref["x_low"] = np.where(same, keep * X.min(axis=0), ref["x_low"])
    ref["x_up"] = np.where(same, keep * X.max(axis=0), ref["x_up"])
    ref["loss0"], ref["loss"] = np.where(same, 0.0, ref["loss0"]), np.where(same, 0.0, ref["loss"])
    assert np.all(np.abs(lo - ref["x_low"]) <= 1e-6 * span + 1e-7 * np.abs(ref["x_low"]) + 1e-45)
    assert np.all(np.abs(hi - ref["x_up"]) <= 1e-6 * span + 1e-7 * np.abs(ref["x_up"]) + 1e-45)
    floor = 1e-12 * n * span ** 2
    assert np.all(np.abs(loss[:D] - ref["loss0"]) <= 1e-9 * ref["loss0"] + floor)
    assert np.all(np.abs(loss[D:] - ref["loss"]) <= 1e-5 * ref["loss"] + floor)


@pytest.mark.parametrize("n,bits", [(1, 4), (5, 4), (9, 4), (64, 4), (1031, 4), (4098, 4), (22528, 4), (22529, 4), (513, 6)])
def test_dual_clip_of_crowded_channels(n, bits):
    X = _channels(n, np.random.default_rng(n))
    _check_against_oracle(X, *_run(X, bits, iters=32, alpha0=6.0), bits)


@pytest.mark.parametrize("D", [300, 640, 1200, 3108, 3256])
def test_crowded_channels_at_every_number_of_warps(D):
    """8, 4, 2, 1 and 1 warps per channel; 1031 values take buckets of two, and of four and eight where 21 or 22 channels share an SM (a
    channel more with the larger buckets).  Equal channels have equal results wherever they stand."""
    X = _channels(1031, np.random.default_rng(D))
    at = np.arange(D) % X.shape[1]
    lo, hi, loss = _run(np.ascontiguousarray(X[:, at]), 4, iters=32, alpha0=6.0)
    for got in (lo, hi, loss[:D], loss[D:]):
        assert np.array_equal(got, got[:X.shape[1]][at])
    few = X.shape[1]
    _check_against_oracle(X, lo[:few], hi[:few], np.concatenate([loss[:few], loss[D:D + few]]), 4)


@pytest.mark.parametrize("n", [33, 2000, 12000])
def test_dual_clip_of_values_far_apart(n):
    """Channels that linear buckets do not part: outliers of every size, two narrow clusters, quartiles that coincide, values that repeat
    around a long tail, a tail on each side over 60 binary orders."""
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 9)).astype(np.float32)
    X[3, 0], X[5, 1], X[7, 2], X[9, 2] = 100.0, 1e6, -1e20, 1e25
    X[:, 3] = np.where(np.arange(n) % 2 == 0, -5.0, 5.0) + 1e-4 * X[:, 3]
    X[:, 4] = np.where(rng.random(n) < 0.7, 0.25, X[:, 4])
    X[:, 5] = np.round(np.exp(2.0 * X[:, 5]))
    X[:, 6] = np.exp(14.0 * X[:, 6]) * np.sign(X[:, 7])
    X[:, 7] = np.sort(X[:, 7])
    X[:, 8] = np.where(np.arange(n) < 3, 1e4, 1.0 + 1e-6 * X[:, 8])
    _check_against_oracle(X, *_run(X, 4, iters=32, alpha0=6.0), 4)


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


def _objective(X, alpha0, Q=15.0):
    """Objective at the starting bounds in 80-bit floats, and what float64 quotients x / s leave open: an error of a few ulp in each
    quotient u, shared through s, moves (q - z - u)^2 by twice its distance."""
    keep = 1.0 / (1.0 + np.exp(-alpha0))
    up, low = X.max(axis=0).astype(np.float64) * keep, X.min(axis=0).astype(np.float64) * keep
    s = (up - low) / Q
    z = np.rint(-low / s)
    u = X.astype(np.longdouble) / s.astype(np.longdouble)
    d = np.clip(np.rint(u), -z, Q - z) - u
    return (s * s * (d * d).sum(axis=0)).astype(np.float64), (2.0 ** -50 * s * s * (2.0 * np.abs(d * u) + d * d).sum(axis=0)).astype(np.float64)


@pytest.mark.parametrize("alpha0", [6.0, 3.0, 2.0, 0.0, -3.0])
def test_objective_is_as_exact_as_float64_values(alpha0):
    """Far outliers on either side, values that lie beyond one of their bounds from the start, two clusters."""
    rng = np.random.default_rng(5)
    X = rng.standard_normal((20001, 9)).astype(np.float32)
    X[7, 1], X[7, 2], X[7, 3], X[9, 4] = -3000.0, 3000.0, -60.0, -3e4
    X[:, 5] = 10.0 - np.abs(X[:, 5]) ** 0.3
    X[:, 6] = np.where(np.arange(len(X)) % 100 == 0, -8.0, 10.0) + 0.2 * X[:, 6]
    X[:, 7] = -np.exp(3.0 * X[:, 7])
    lo, hi, loss = _run(X, 4, iters=100, alpha0=alpha0)
    exact, open_ = _objective(X, alpha0)
    assert np.all(np.abs(loss[:9] - exact) <= open_), np.abs(loss[:9] - exact) / open_
    # (a channel that lies beyond one of its bounds steps back and forth over the jumps of its zero point: the order of the sums alone
    # then moves the bounds by per cent; such channels are told by the oracle's own answer to the rows in reverse)
    from oracle import repq_oracle as orc
    ref, again = (orc.dual_clip(x, 4, iters=100, lr=0.01, alpha0=alpha0) for x in (X, X[::-1]))
    span = X.max(axis=0).astype(np.float64) - X.min(axis=0)
    settled = np.maximum(np.abs(ref["x_low"] - again["x_low"]), np.abs(ref["x_up"] - again["x_up"])) <= 1e-9 * span
    assert settled.sum() >= 8
    assert np.all((np.abs(lo - ref["x_low"]) <= 1e-6 * span)[settled]) and np.all((np.abs(hi - ref["x_up"]) <= 1e-6 * span)[settled])
