"""The activation-derivative epilogue of the backward (du, dv and the row dots) at the edges
of its 16-column steps, 32-column chunks and 128-row halves: widths below, at and past a
chunk, widths that are no multiple of 8, tiles with one row more or less than a half.
Every gradient against the oracle's backward, tolerances as for the layer."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2608_17402_gb300 import moevie
from tests._gpu import assert_close, check_status, dev, dev_bf16, layer_to_device, to_np_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("act", ["gelu", "swiglu"])
@pytest.mark.parametrize("T,h,hs", [(40, 8, 0), (127, 16, 0), (128, 31, 0), (129, 33, 0), (65, 63, 0), (257, 65, 40),
                                    (30, 250, 0), (300, 264, 300)])
def test_backward_widths(T, h, hs, act):
    d, E, k = 72, 5, 2
    cfg = workloads.small_config(T, d, E, k, h, h_s=hs, lam=0.5 if hs else 1.0, seed=T + h, act=act)
    lay = workloads.make_layer(cfg)
    rng = np.random.default_rng(h)
    dy_bits = workloads.f32_to_bf16_bits(rng.standard_normal((T, d)).astype(np.float32))
    idx, _, _ = oracle.route(lay.x, lay.Wr, lay.b, k)
    extra = {"W3": lay.W3} if act == "swiglu" else {}
    if hs:
        extra.update(Ws1=lay.Ws1, Ws2=lay.Ws2, lam=cfg.lam)
        if act == "swiglu":
            extra["Ws3"] = lay.Ws3
    want = oracle.backward(lay.x, lay.Wr, lay.b, lay.W1, lay.W2, k,
                           workloads.bf16_bits_to_f32(dy_bits).astype(np.float64), **extra)
    x, W = layer_to_device(lay)
    ws = moevie.BackwardWorkspace(T, d, E, k, h, h_s=hs, swiglu=act == "swiglu")
    got = moevie.moevie_moe_backward(W, x, dev_bf16(dy_bits), dev(np.ascontiguousarray(idx, np.int32)), ws)
    check_status(ws)
    for name, ref in [("dx", "dx"), ("dW_r", "dWr")] + [(n, n) for n in ("dW1", "dW2", "dW3", "dWs1", "dWs2", "dWs3")
                                                        if n in got]:
        assert_close(to_np_f64(got[name]), want[ref], name)
