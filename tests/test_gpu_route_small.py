"""The one-launch router (small tokens x experts x d) at its edges: token counts around its
8 tokens a CTA and its largest, experts around the 32 of a lane slot, d around its slices
and chunks up to its largest, and inputs that send tokens to the exact re-decision.  Ids equal to the oracle's, gates within 1e-5, as for the other route."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2608_17402_gb300 import moevie
from tests._gpu import MARGIN_PINNED, check_status, dev, dev_bf16

pytestmark = pytest.mark.gpu


def _check(x, Wr, b, k):
    T, d = x.shape
    ws = moevie.Workspace(T, d, Wr.shape[1], k, 16)
    n0 = moevie.moevie_launch_count()
    for _ in range(2):   # the counters in the workspace are left ready for the next call
        idx, gate = moevie.moevie_route(dev_bf16(x), dev(Wr), dev(b), k, ws)
    check_status(ws)
    assert moevie.moevie_launch_count() - n0 == 2, "these sizes take one launch"
    nfb = moevie.moevie_test_fallback_count(ws)
    oidx, ogate, margin = oracle.route(x, Wr, b, k)
    pinned = margin > MARGIN_PINNED
    assert np.array_equal(idx.cpu().numpy()[pinned], oidx[pinned])
    np.testing.assert_allclose(gate.cpu().numpy()[pinned], ogate[pinned], rtol=0, atol=1e-5)
    return nfb


def _inputs(T, d, E, seed):
    rng = np.random.default_rng(seed)
    x = workloads.f32_to_bf16_bits(rng.standard_normal((T, d)).astype(np.float32))
    Wr = (rng.standard_normal((d, E)) * 0.02).astype(np.float32)
    return x, Wr, rng.uniform(-0.1, 0.1, E).astype(np.float32)


@pytest.mark.parametrize("T,d,E,k", [
    (1, 8, 1, 1), (3, 16, 2, 1), (7, 24, 31, 3), (8, 64, 32, 8), (9, 72, 33, 4), (17, 264, 64, 8), (33, 512, 63, 8),
    (40, 136, 48, 8), (16, 1024, 32, 8), (1215, 40, 16, 2), (1216, 1024, 20, 3), (1209, 512, 64, 8), (6, 32, 8, 8),
])
def test_small_router_edges(T, d, E, k):
    _check(*_inputs(T, d, E, T + d + E), k)


@pytest.mark.parametrize("T,E", [(50, 24), (1200, 48), (1111, 33)])
def test_small_router_ties_go_to_the_exact_decision(T, E):
    x, Wr, b = _inputs(T, 96, E, T)
    Wr[:, 1::2] = Wr[:, : 2 * (E // 2) : 2]   # every even expert has a twin: exact ties
    b[1::2] = b[: 2 * (E // 2) : 2]
    ws_fb = _ties(x, Wr, b, 3)
    assert ws_fb > 0


def _ties(x, Wr, b, k):
    T, d = x.shape
    ws = moevie.Workspace(T, d, Wr.shape[1], k, 16)
    idx, gate = moevie.moevie_route(dev_bf16(x), dev(Wr), dev(b), k, ws)
    check_status(ws)
    oidx, ogate, _ = oracle.route(x, Wr, b, k)
    assert np.array_equal(idx.cpu().numpy(), oidx)   # equal sums in any order: ties stay ties
    np.testing.assert_allclose(gate.cpu().numpy(), ogate, rtol=0, atol=1e-5)
    return moevie.moevie_test_fallback_count(ws)


def test_small_router_wide_range_of_magnitudes():
    """Weights over many binades and cancelling rows: the error bound and the exact window."""
    x, Wr, b = _inputs(64, 128, 40, 3)
    rng = np.random.default_rng(4)
    Wr *= np.exp2(rng.integers(-40, 6, Wr.shape)).astype(np.float32)
    _check(x, Wr, b, 4)
