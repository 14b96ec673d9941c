"""The transposed product behind the down-projection and the backward's dx (rows reduced
into their tokens' rows of an fp32 accumulator) at the edges of its tiles: the MMA's N is
the tile's rows rounded up to 64, its M 256 output columns, 128 per CTA, 32 per warp.
With W_r = 0 every token selects the k experts of largest bias, so each of them holds
exactly T rows.  Tolerances are the layer's (bf16 operands, fp32 accumulation)."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2608_17402_gb300 import moevie
from tests._gpu import assert_close, check_status, dev, dev_bf16, layer_to_device, to_np_f64, workspace_for

pytestmark = pytest.mark.gpu


def _layer(T, d, h, hs=0):
    cfg = workloads.small_config(T, d, 5, 2, h, h_s=hs, lam=0.5 if hs else 1.0, seed=T + d + h)
    lay = workloads.make_layer(cfg)
    lay.Wr[:] = 0.0
    return lay


ROWS = [1, 31, 32, 33, 63, 64, 65, 128, 129, 191, 192, 193, 255, 256, 257, 321]
COLS = [8, 120, 128, 136, 256, 264, 520]


@pytest.mark.parametrize("T,d,hs", [(T, 136, 0) for T in ROWS] + [(70, d, 0) for d in COLS] + [(200, 264, 64)])
def test_down_projection_tiles(T, d, hs):
    lay = _layer(T, d, 64, hs)
    x, W = layer_to_device(lay)
    ws = workspace_for(lay)
    y = to_np_f64(moevie.moevie_moe_forward(W, x, ws))
    check_status(ws)
    want, *_ = oracle.forward_tokens(lay.x, lay.Wr, lay.b, lay.W1, lay.W2, 2, lay.Ws1, lay.Ws2, lay.cfg.lam)
    assert_close(y, want)


@pytest.mark.parametrize("T,d,h", [(1, 136, 40), (64, 136, 64), (65, 256, 40), (129, 264, 72), (257, 120, 64)])
def test_backward_dx_tiles(T, d, h):
    lay = _layer(T, d, h)
    rng = np.random.default_rng(T)
    dy_bits = workloads.f32_to_bf16_bits(rng.standard_normal((T, d)).astype(np.float32))
    idx, _, _ = oracle.route(lay.x, lay.Wr, lay.b, 2)
    want = oracle.backward(lay.x, lay.Wr, lay.b, lay.W1, lay.W2, 2,
                           workloads.bf16_bits_to_f32(dy_bits).astype(np.float64))
    x, W = layer_to_device(lay)
    ws = moevie.BackwardWorkspace(T, d, 5, 2, h)
    got = moevie.moevie_moe_backward(W, x, dev_bf16(dy_bits), dev(np.ascontiguousarray(idx, np.int32)), ws)
    check_status(ws)
    assert_close(to_np_f64(got["dx"]), want["dx"])
