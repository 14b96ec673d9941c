"""Tokens whose keys tie, or nearly do, through the one-launch router (small tokens x experts x d):
every candidate count, expert count and width its exact sums are split differently for, logits
whose rounding errors exceed the gaps between them, and the time such calls may take."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from paper_2608_17402_gb300 import moevie
from tests._gpu import MARGIN_PINNED, check_status, dev, dev_bf16

pytestmark = pytest.mark.gpu


def _route(x, Wr, b, k):
    """ids, gates and the number of re-decided tokens of one call, which takes one launch."""
    ws = moevie.Workspace(x.shape[0], x.shape[1], Wr.shape[1], k, 16)
    n0 = moevie.moevie_launch_count()
    idx, gate = moevie.moevie_route(dev_bf16(x), dev(Wr), dev(b), k, ws)
    check_status(ws)
    assert moevie.moevie_launch_count() - n0 == 1
    return idx.cpu().numpy(), gate.cpu().numpy(), moevie.moevie_test_fallback_count(ws)


@pytest.mark.parametrize("T,d,E,k", [
    (1, 8, 5, 2), (8, 24, 8, 3), (9, 1024, 8, 7), (17, 264, 9, 4), (8, 1024, 16, 2), (33, 136, 17, 16), (16, 1024, 32, 8),
    (7, 512, 33, 8), (25, 504, 64, 63), (1216, 512, 64, 8),
])
def test_every_key_ties(T, d, E, k):
    """Equal columns and biases: the k lowest ids, gates 1 / k."""
    rng = np.random.default_rng(T + d + E)
    x = workloads.f32_to_bf16_bits(rng.standard_normal((T, d)).astype(np.float32))
    Wr = np.repeat((rng.standard_normal((d, 1)) * 0.02).astype(np.float32), E, axis=1)
    idx, gate, nfb = _route(x, Wr, np.zeros(E, np.float32), k)
    assert nfb == T
    assert np.array_equal(idx, np.tile(np.arange(k), (T, 1)))
    np.testing.assert_allclose(gate, 1.0 / k, rtol=0, atol=1e-6)


@pytest.mark.parametrize("n", [2, 4, 5, 9])
@pytest.mark.parametrize("d,E", [(1024, 31), (256, 12), (512, 60)])
def test_groups_of_equal_experts(n, d, E):
    """Groups of n equal experts among others: ties at the boundary with about n candidates."""
    rng = np.random.default_rng(n * E)
    T, k = 100, 4
    x = workloads.f32_to_bf16_bits(rng.standard_normal((T, d)).astype(np.float32))
    col = np.arange(E) // n
    Wr = (rng.standard_normal((d, E)) * 0.02).astype(np.float32)[:, col]
    b = rng.uniform(-0.01, 0.01, E).astype(np.float32)[col]
    perm = rng.permutation(E)
    Wr, b = np.ascontiguousarray(Wr[:, perm]), b[perm]
    idx, gate, nfb = _route(x, Wr, b, k)
    oidx, ogate, _ = oracle.route(x, Wr, b, k)
    assert k % n == 0 or nfb > T // 4   # the boundary falls inside a group
    assert np.array_equal(idx, oidx)
    np.testing.assert_allclose(gate, ogate, rtol=0, atol=1e-5)


@pytest.mark.parametrize("T", [152, 153, 305, 460, 610, 913, 1216])
@pytest.mark.parametrize("d,E,some", [(200, 24, 1), (512, 40, 3)])
def test_pairs_of_equal_experts_on_many_tokens(T, d, E, some):
    """One to eight tokens a CTA, all of them (or every third) with two or four candidates for
    the last place: odd k splits a pair of equal experts."""
    rng = np.random.default_rng(T + E)
    k = 3
    xf = rng.standard_normal((T, d)).astype(np.float32)
    xf[:, 0] = (np.arange(T) % some != 0) * 8.0     # moves the pairs apart on the other tokens
    x = workloads.f32_to_bf16_bits(xf)
    Wr = np.repeat((rng.standard_normal((d, E // 2)) * 0.02).astype(np.float32), 2, axis=1)
    Wr[0, 1::2] += 0.05
    b = np.repeat(rng.uniform(-0.1, 0.1, E // 2).astype(np.float32), 2)
    b[2:4] = b[0:2]
    Wr[:, 2:4] = Wr[:, 0:2]                         # and one group of four
    idx, gate, nfb = _route(x, Wr, b, k)
    oidx, ogate, _ = oracle.route(x, Wr, b, k)
    assert nfb >= T // some
    assert np.array_equal(idx, oidx)
    np.testing.assert_allclose(gate, ogate, rtol=0, atol=1e-5)


@pytest.mark.parametrize("pattern", ["halves", "alternating", "slices"])
@pytest.mark.parametrize("d,E", [(1024, 32), (512, 64), (776, 31)])
def test_rounding_errors_larger_than_the_gaps(pattern, d, E):
    """Products of about 100 that cancel exactly (the partial sums growing to half of all, not at
    all, or within each warp's slice of d) beside 64 ordinary ones: the fp32 sums are off by far
    more than the gaps between the experts and than the slack of the keys, so only a certificate
    whose bound covers the whole error leaves these tokens to the exact sums."""
    rng = np.random.default_rng(d + E)
    T, k, m = 64, 6, (d - 64) // 16 * 16
    sign = {"halves": np.repeat([1.0, -1.0], m // 2), "alternating": np.tile([1.0, -1.0], m // 2),
            "slices": np.tile(np.repeat([1.0, -1.0], 8), m // 16)}[pattern]
    xf = rng.standard_normal((T, d)).astype(np.float32)
    xf[:, :m] = 1.0
    x = workloads.f32_to_bf16_bits(xf)
    Wr = (rng.standard_normal((d, E)) * 0.05).astype(np.float32)
    base = 100.0 * (1.0 + rng.uniform(0.0, 2.0 ** -4, (m, E)))
    base[sign < 0] = base[sign > 0]        # the same magnitudes with either sign
    Wr[:m] = (sign[:, None] * base).astype(np.float32)
    b = rng.uniform(-0.01, 0.01, E).astype(np.float32)
    idx, _, nfb = _route(x, Wr, b, k)
    oidx, _, margin = oracle.route(x, Wr, b, k)
    pinned = margin > MARGIN_PINNED
    assert pinned.mean() > 0.99
    assert nfb > T // 2
    assert np.array_equal(idx[pinned], oidx[pinned])


def _time_us(T, d, E, k):
    """One call of moevie_route on tokens that all tie (W_r = 0, b = 0), back to back calls."""
    x = torch.randn((T, d), device="cuda").to(torch.bfloat16)
    Wr, b = torch.zeros((d, E), device="cuda"), torch.zeros(E, device="cuda")
    ws = moevie.Workspace(T, d, E, k, 16)
    idx = torch.zeros((T, k), dtype=torch.int32, device="cuda")
    gate = torch.zeros((T, k), device="cuda")
    best = float("inf")
    for _ in range(6):
        a, c = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            moevie.moevie_route(x, Wr, b, k, ws, idx, gate)
        c.record()
        c.synchronize()
        best = min(best, a.elapsed_time(c) / 20 * 1e3)
    return best


@pytest.mark.parametrize("small,large", [
    ((1216, 1024, 32, 8), (1217, 1024, 32, 8)), ((1216, 512, 64, 8), (1217, 512, 64, 8)), ((64, 1024, 32, 8), (64, 1032, 32, 8)),
    ((256, 1024, 31, 3), (256, 1032, 31, 3)), ((512, 1024, 16, 2), (512, 1032, 16, 2)), ((16, 512, 64, 8), (16, 520, 64, 8)),
])
def test_ties_cost_no_more_than_on_the_other_route(small, large):
    """The one-launch router on tokens that all tie against the tensor-core route at the next size
    past the line between them (a tenth for the spread of the clocks)."""
    a, b = _time_us(*small), _time_us(*large)
    print(f"{small}: {a:.1f} us, {large}: {b:.1f} us")
    assert a <= 1.1 * b, (small, a, large, b)
