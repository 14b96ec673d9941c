"""The two forms of an accumulating GEMM (down-projection, the backward's dx) on both sides of the
rule between them: the transposed product, and with many rows a group on few columns past a
multiple of 256 the staged one.  Oracle and tolerance of the layer."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2608_17402_gb300 import moevie
from tests._gpu import assert_close, check_status, dev, dev_bf16, layer_to_device, to_np_f64, workspace_for

pytestmark = pytest.mark.gpu

# rows a group r = T / E; staged: r above 5 at 64 columns, 85 at 128, 179 at 264, 420 at 520, any at 8
SHAPES = [(130, 8, 3, 16), (40, 64, 2, 40), (700, 64, 2, 40), (300, 128, 2, 64), (340, 264, 2, 72), (380, 264, 2, 72),
          (700, 320, 2, 40), (820, 520, 2, 40), (900, 520, 2, 100), (900, 512, 2, 40), (700, 776, 2, 40)]


def _layer(T, d, E, h, act):
    lay = workloads.make_layer(workloads.small_config(T, d, E, 1, h, seed=T + d, act=act))
    return lay, *layer_to_device(lay)


@pytest.mark.parametrize("act", ["gelu", "swiglu"])
@pytest.mark.parametrize("T,d,E,h", SHAPES)
def test_down_projection_forms(T, d, E, h, act):
    lay, x, W = _layer(T, d, E, h, act)
    ws = workspace_for(lay)
    y = to_np_f64(moevie.moevie_moe_forward(W, x, ws))
    check_status(ws)
    want, *_ = oracle.forward_tokens(lay.x, lay.Wr, lay.b, lay.W1, lay.W2, 1, W3=lay.W3)
    assert_close(y, want)


@pytest.mark.parametrize("act", ["gelu", "swiglu"])
@pytest.mark.parametrize("T,d,E,h", SHAPES)
def test_dx_forms(T, d, E, h, act):
    lay, x, W = _layer(T, d, E, h, act)
    dy_bits = workloads.f32_to_bf16_bits(np.random.default_rng(T).standard_normal((T, d)).astype(np.float32))
    idx, _, _ = oracle.route(lay.x, lay.Wr, lay.b, 1)
    want = oracle.backward(lay.x, lay.Wr, lay.b, lay.W1, lay.W2, 1, workloads.bf16_bits_to_f32(dy_bits).astype(np.float64), W3=lay.W3)
    ws = moevie.BackwardWorkspace(T, d, E, 1, h, swiglu=act == "swiglu")
    got = moevie.moevie_moe_backward(W, x, dev_bf16(dy_bits), dev(np.ascontiguousarray(idx, np.int32)), ws)
    check_status(ws)
    assert_close(to_np_f64(got["dx"]), want["dx"])
