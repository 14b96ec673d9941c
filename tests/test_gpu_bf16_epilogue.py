"""The bf16 epilogue of the grouped up-projection (rows in 32s, columns in 32s through shared memory)
at the edges of its tiles: experts of 0, 1, 31 .. 257 rows, widths around 8, 32 and 256 columns, K from
one partial block on.  Reference in fp64; each element may be off by the fp32 sum of d products
(d 2^-24 sum |x w|, through GELU' <= 1.13), the GELU's 1e-6 and half a bf16 unit."""
import numpy as np
import pytest
import torch

import workloads
from paper_2608_17402_gb300 import moevie
from tests._gpu import check_status, dev, dev_bf16, dev_rows, to_np_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [(1, 0, 31), (32, 33, 127), (128, 129, 255), (256, 257, 5)])
@pytest.mark.parametrize("d,h", [(8, 8), (64, 36), (72, 100), (512, 264), (1032, 520)])
def test_expert_hidden_edges(counts, d, h):
    rng = np.random.default_rng(sum(counts) + d + h)
    E, T = len(counts), sum(counts)
    x = workloads.f32_to_bf16_bits(rng.standard_normal((T, d)).astype(np.float32))
    W1 = workloads.f32_to_bf16_bits((rng.standard_normal((E, d, h)) * d ** -0.5).astype(np.float32))
    perm = rng.permutation(T).astype(np.int32)
    offsets = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    ws = moevie.Workspace(T, d, E, 1, h)
    got = to_np_f64(moevie.moevie_test_expert_hidden(dev_bf16(x), dev(perm), dev(offsets), dev_rows(W1), 1, ws))
    check_status(ws)
    xf = torch.from_numpy(workloads.bf16_bits_to_f32(x).astype(np.float64))[torch.from_numpy(perm.astype(np.int64))]
    wf = torch.from_numpy(workloads.bf16_bits_to_f32(W1).astype(np.float64))
    for e in range(E):
        r = slice(int(offsets[e]), int(offsets[e + 1]))
        want = torch.nn.functional.gelu(xf[r] @ wf[e]).numpy()
        err = 1.13 * d * 2.0 ** -24 * (xf[r].abs() @ wf[e].abs()).numpy() + 1e-6
        half_unit = np.exp2(np.floor(np.log2(np.abs(want) + err)) - 8)   # bf16: eight significant bits
        assert np.all(np.abs(got[r, :h] - want) <= err + half_unit), (e, counts, d, h)
