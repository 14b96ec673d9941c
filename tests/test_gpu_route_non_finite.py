"""Infinities and NaN in the router's inputs, on both routes: every token still gets k different ids in
ascending order inside [0, E), nothing is written past its k slots, and the tokens whose own
inputs are finite get what they get alone."""
import numpy as np
import pytest
import torch

from paper_2608_17402_gb300 import moevie
from tests._gpu import check_status

pytestmark = pytest.mark.gpu

SIZES = [(40, 64, 16, 3), (33, 64, 40, 5), (1300, 64, 16, 3), (40, 64, 100, 7), (40, 1032, 31, 8)]   # one launch, one, four ...
GUARD = 64


def _route(x, W, b, k):
    T, E = x.shape[0], W.shape[1]
    ws = moevie.Workspace(T, x.shape[1], E, k, 16)
    idx = torch.full((T + GUARD, k), -7, dtype=torch.int32, device="cuda")
    gate = torch.full((T + GUARD, k), -7.0, device="cuda")
    moevie.moevie_route(x, W, b, k, ws, idx[:T], gate[:T])
    check_status(ws)
    assert bool((idx[T:] == -7).all()) and bool((gate[T:] == -7.0).all())
    i = idx[:T].cpu().numpy()
    assert i.min() >= 0 and i.max() < E and (k == 1 or np.all(np.diff(i, axis=1) > 0))
    return i, gate[:T].cpu().numpy()


def _inputs(T, d, E):
    g = torch.Generator(device="cuda")
    g.manual_seed(T + E)
    return (torch.randn((T, d), generator=g, device="cuda"), torch.randn((d, E), generator=g, device="cuda") * 0.02,
            torch.rand(E, generator=g, device="cuda") * 0.2)


@pytest.mark.parametrize("T,d,E,k", SIZES)
def test_tokens(T, d, E, k):
    x, W, b = _inputs(T, d, E)
    want, gates = _route(x.bfloat16(), W, b, k)
    bad = [3, 4, 5, 6, T - 1]
    x[3, 5], x[4, 6], x[5, 7], x[T - 1, 0] = float("inf"), float("nan"), float("-inf"), float("nan")
    x[6, 1:3] = float("inf")
    idx, gate = _route(x.bfloat16(), W, b, k)
    ok = np.setdiff1d(np.arange(T), bad)
    assert np.array_equal(idx[ok], want[ok]) and np.array_equal(gate[ok], gates[ok])


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("T,d,E,k", SIZES)
def test_experts(T, d, E, k, value):
    x, W, b = _inputs(T, d, E)
    W[3, 2], W[4, E - 1] = value, value
    _route(x.bfloat16(), W, b, k)
    x, W, b = _inputs(T, d, E)
    b[2], b[5] = value, -value
    _route(x.bfloat16(), W, b, k)
