"""The permute over one cluster of eight CTAs (at most 2048 slots): slot counts around its
chunks of 256 slots, CTAs without slots, and its largest count; beside them the first count
that takes the grid-wide kernel.  Every output equal to the oracle's, also in a workspace of
exactly the size asked for, and the by-products of a forward that does not ask for them."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from paper_2608_17402_gb300 import moevie
from tests._gpu import check_status, dev, layer_to_device, workspace_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,E,k", [
    (1, 3, 1), (255, 5, 1), (256, 5, 1), (257, 5, 1), (768, 31, 1), (2047, 64, 1), (2048, 64, 1), (2049, 1024, 1),
    (255, 64, 8), (256, 64, 8), (256, 1024, 8), (300, 64, 8), (1500, 7, 1),
])
def test_permute_cluster(T, E, k):
    rng = np.random.default_rng(T + E)
    idx = np.stack([np.sort(rng.choice(E, size=k, replace=False)) for _ in range(T)]).astype(np.int32)
    ws = moevie.Workspace(T, 8, E, k, 16)
    for _ in range(2):   # nothing is left behind between calls
        counts, offsets, perm, inv = moevie.moevie_permute(dev(idx), E, ws)
    check_status(ws)
    oc, oo, op, oi = oracle.permute(idx, E)
    assert np.array_equal(counts.cpu().numpy(), oc)
    assert np.array_equal(offsets.cpu().numpy(), oo)
    assert np.array_equal(perm.cpu().numpy(), op)
    assert np.array_equal(inv.cpu().numpy(), oi)
    c2 = moevie.moevie_permute_static(dev(idx), E)
    for a, b in zip(c2, (counts, offsets, perm, inv)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("T", [40, 1100])
def test_forward_with_and_without_by_products(T):
    lay = workloads.make_layer(workloads.small_config(T, 64, 9, 8, 40, seed=T))
    x, W = layer_to_device(lay)
    ws = workspace_for(lay)
    y, rt = moevie.moevie_moe_forward(W, x, ws, routing=True)
    y2 = moevie.moevie_moe_forward(W, x, ws)
    check_status(ws)
    _, _, op, oi = oracle.permute(rt["idx"].cpu().numpy(), 9)
    assert np.array_equal(rt["perm"].cpu().numpy(), op) and np.array_equal(rt["inv"].cpu().numpy(), oi)
    # the same rows in the same tiles; fp32 sums of eight experts may differ in their order
    torch.testing.assert_close(y2.float(), y.float(), rtol=2.0 ** -7, atol=1e-3)
