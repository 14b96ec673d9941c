"""The backward's per-token kernels (gates, router) at every selection width they are compiled
for and past it: k = 1 .. 8 have their own, more go in passes of 8.  Compared are the gradients
they form, of x and of W_r, with the oracle and the tolerance of the other backward tests."""
import numpy as np
import pytest

import oracle
import workloads
from tests._gpu import assert_close
from tests.test_gpu_backward import _dy, _gpu_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,E,k", [
    (65, 72, 40, 1), (65, 72, 40, 2), (65, 136, 40, 3), (65, 72, 40, 4), (65, 72, 40, 5), (65, 136, 40, 6), (65, 264, 40, 7),
    (65, 72, 40, 8), (70, 200, 40, 9), (33, 72, 16, 16), (70, 328, 40, 17), (70, 64, 33, 24), (70, 136, 64, 31), (70, 264, 32, 32),
])
def test_backward_selection_widths(T, d, E, k):
    lay = workloads.make_layer(workloads.small_config(T, d, E, k, 64, seed=T + d + k))
    dy_bits, dyf = _dy(T, d, k)
    idx, _, _ = oracle.route(lay.x, lay.Wr, lay.b, k)
    want = oracle.backward(lay.x, lay.Wr, lay.b, lay.W1, lay.W2, k, dyf)
    got = _gpu_backward(lay, dy_bits, idx)
    assert_close(got["dx"], want["dx"], "dx")
    if k > 1:
        assert_close(got["dW_r"], want["dWr"], "dW_r")
    else:   # one gate, always 1
        assert not np.any(got["dW_r"])


def test_backward_bad_ids_are_dropped_at_any_width():
    """An id outside [0, E) is reported and adds nothing; the other slots' results stay finite."""
    from paper_2608_17402_gb300 import moevie
    from tests._gpu import dev, dev_bf16, layer_to_device
    T, d, E, k = 40, 72, 24, 11
    lay = workloads.make_layer(workloads.small_config(T, d, E, k, 64, seed=3))
    idx, _, _ = oracle.route(lay.x, lay.Wr, lay.b, k)
    idx = np.ascontiguousarray(idx, np.int32)
    idx[5, 10], idx[7, 2] = E, -1
    dy_bits, _ = _dy(T, d, 4)
    x, W = layer_to_device(lay)
    ws = moevie.BackwardWorkspace(T, d, E, k, 64)
    g = moevie.moevie_moe_backward(W, x, dev_bf16(dy_bits), dev(idx), ws)
    code, _ = moevie.moevie_get_device_status(ws)
    assert code != 0
    assert all(bool(v.isfinite().all()) for v in g.values())
