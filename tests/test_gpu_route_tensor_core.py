"""The tensor-core route (split of W_r, GEMM, top-k, exact re-decision) on sizes past the one-launch
router's: ragged token counts on either layout of the two pieces (side by side up to E = 128),
exact ties, cancelling, tiny and subnormal weights, and a selection by the bias alone."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2608_17402_gb300 import moevie
from tests._gpu import MARGIN_PINNED, check_status, dev, dev_bf16

pytestmark = pytest.mark.gpu


def _route(x, Wr, b, k):
    """ids, gates and the number of re-decided tokens of one call, which takes four launches."""
    ws = moevie.Workspace(x.shape[0], x.shape[1], Wr.shape[1], k, 16)
    n0 = moevie.moevie_launch_count()
    idx, gate = moevie.moevie_route(dev_bf16(x), dev(Wr), dev(b), k, ws)
    check_status(ws)
    assert moevie.moevie_launch_count() - n0 == 4, "these sizes take the tensor-core route"
    return idx.cpu().numpy(), gate.cpu().numpy(), moevie.moevie_test_fallback_count(ws)


def _inputs(T, d, E, std=0.02):
    rng = np.random.default_rng(T + d + E)
    x = workloads.f32_to_bf16_bits(rng.standard_normal((T, d)).astype(np.float32))
    return rng, x, (rng.standard_normal((d, E)) * std).astype(np.float32), rng.uniform(-0.1, 0.1, E).astype(np.float32)


@pytest.mark.parametrize("T,d,E,k", [
    (1217, 16, 8, 2), (1301, 64, 16, 2), (1217, 96, 1, 1), (1500, 32, 4, 4), (1217, 48, 33, 5), (1301, 128, 64, 8),
    (1, 1032, 8, 2), (129, 1032, 32, 8), (77, 520, 48, 5), (37, 24, 65, 3), (300, 104, 100, 8), (257, 64, 128, 8), (513, 40, 129, 4),
])
def test_ragged_sizes(T, d, E, k):
    _, x, Wr, b = _inputs(T, d, E)
    idx, gate, _ = _route(x, Wr, b, k)
    oidx, ogate, margin = oracle.route(x, Wr, b, k)
    pinned = margin > MARGIN_PINNED
    assert pinned.mean() > 0.999
    assert np.array_equal(idx[pinned], oidx[pinned])
    np.testing.assert_allclose(gate[pinned], ogate[pinned], rtol=0, atol=1e-5)


@pytest.mark.parametrize("T,d,E,k", [(1301, 64, 16, 3), (256, 1032, 31, 3), (200, 520, 60, 7), (128, 64, 100, 5), (100, 48, 300, 9)])
def test_ties_go_to_the_lower_id(T, d, E, k):
    """Every even expert has a twin of equal column and bias: odd k splits pairs."""
    _, x, Wr, b = _inputs(T, d, E, 0.3)
    Wr[:, 1::2] = Wr[:, : 2 * (E // 2) : 2]
    b[1::2] = b[: 2 * (E // 2) : 2]
    idx, gate, nfb = _route(x, Wr, b, k)
    oidx, ogate, _ = oracle.route(x, Wr, b, k)
    assert nfb > T // 2
    assert np.array_equal(idx, oidx)
    np.testing.assert_allclose(gate, ogate, rtol=0, atol=1e-5)


@pytest.mark.parametrize("T,d,E,k", [(1301, 64, 24, 4), (64, 1032, 32, 8), (64, 40, 130, 5)])
def test_every_key_ties(T, d, E, k):
    _, x, Wr, _ = _inputs(T, d, E)
    idx, gate, nfb = _route(x, np.repeat(Wr[:, :1], E, axis=1), np.zeros(E, np.float32), k)
    assert nfb == T
    assert np.array_equal(idx, np.tile(np.arange(k), (T, 1)))
    np.testing.assert_allclose(gate, 1.0 / k, rtol=0, atol=1e-6)


@pytest.mark.parametrize("T,d,E,k", [(1301, 96, 24, 4), (256, 96, 100, 4), (200, 1032, 24, 4)])
def test_exact_sums_of_cancelling_and_tiny_terms(T, d, E, k):
    """Two rows of products that cancel exactly (x[:, 1] = x[:, 0], W_r[1] = -W_r[0] = 1024 r) make the
    error bound of the fast logits large; rows of tiny (2^-40) and subnormal weights fall far
    below the others; a near-duplicate column differs from its twin by x[:, 10] 2^-20 only."""
    rng, x, Wr, b = _inputs(T, d, E, 0.05)
    x[:, 1] = x[:, 0]
    Wr[0] = (1024.0 * rng.uniform(0.5, 1.0, E) * rng.choice([-1.0, 1.0], E)).astype(np.float32)
    Wr[1] = -Wr[0]
    Wr[2:6] *= np.float32(2.0 ** -40)
    Wr[6:10] = (rng.standard_normal((4, E)) * 1e-40).astype(np.float32)
    Wr[:, 17] = Wr[:, 3]
    Wr[10, 17] = Wr[10, 3] + np.float32(2.0 ** -20)
    b[17] = b[3]
    idx, gate, nfb = _route(x, Wr, b, k)
    oidx, ogate, margin = oracle.route(x, Wr, b, k)
    pinned = margin > MARGIN_PINNED
    assert pinned.mean() > 0.99 and nfb > T // 2
    assert np.array_equal(idx[pinned], oidx[pinned])


def test_bias_only():
    """W_r = 0: every key is 1/2 + b; ties in b resolve to the lower id; gates 1/k."""
    T, d, E, k = 1300, 32, 12, 4
    x = workloads.f32_to_bf16_bits(np.random.default_rng(1).standard_normal((T, d)).astype(np.float32))
    b = np.array([0.0625, -0.5, 0.25, 0.25, 0.0, 0.25, 0.125, 0.25, -0.25, 0.0625, 0.5, 0.0], np.float32)
    idx, gate, _ = _route(x, np.zeros((d, E), np.float32), b, k)
    assert np.all(idx == np.array([2, 3, 5, 10]))   # 0.5 (id 10), then 0.25 at ids 2, 3, 5 (7 left out)
    np.testing.assert_allclose(gate, 0.25, rtol=0, atol=1e-7)
