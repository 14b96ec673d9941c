"""The gathered GEMM's A row of a routing slot, slot / k by a multiplication: against the division
itself for every k up to 1024 (the host's constants, on the CPU), and the rows it gathers."""
import subprocess

import numpy as np
import pytest
import torch

import workloads
from paper_2608_17402_gb300 import _build, moevie

PROGRAM = r"""
#include <stdio.h>
#include "internal.h"
int main() {
    const int64_t top = (int64_t(1) << 31) - 1;
    for (int div = 1; div <= 1024; ++div) {
        uint32_t mul;
        int shift;
        mv::div_by_mul(div, &mul, &shift);
        const int64_t last = top / div * div;
        for (int64_t q = 0; q < 4000; ++q) {
            const int64_t base[5] = {q * div, last - q * div, q * 536861 / div * div, top - q, q};
            for (int64_t b : base)
                for (int64_t r = b - 1; r <= b + 1; ++r)
                    if (r >= 0 && r <= top && (int64_t)((uint64_t)r * mul >> shift) != r / div) {
                        printf("%lld / %d\n", (long long)r, div);
                        return 1;
                    }
        }
    }
    return 0;
}
"""


def test_multiplication_equals_the_division(tmp_path):
    src = tmp_path / "div.cu"
    src.write_text(PROGRAM)
    subprocess.run([_build._nvcc(), "-O2", "-std=c++17", "-I", _build.INCLUDE, "-I", _build.CSRC, "--expt-relaxed-constexpr",
                    *_build.ARCH, str(src), "-o", str(tmp_path / "div"), "-lcuda"], check=True, capture_output=True)
    r = subprocess.run([str(tmp_path / "div")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("T,k", [(97, 1), (97, 2), (200, 3), (61, 5), (300, 7), (40, 8), (33, 31), (20, 33), (5, 777), (3, 1024)])
def test_slots_gather_their_tokens(T, k):
    """Hidden rows of slots t k + j are those of k = 1 on the tokens t themselves, bit for bit."""
    from tests._gpu import check_status, dev, dev_bf16, dev_rows
    rng = np.random.default_rng(T * k)
    d, h = 64, 32
    x = dev_bf16(workloads.f32_to_bf16_bits(rng.standard_normal((T, d)).astype(np.float32)))
    W1 = dev_rows(workloads.f32_to_bf16_bits(rng.standard_normal((1, d, h)).astype(np.float32)))
    W1 = W1.expand(1, d, h) if k == 1 else moevie.moevie_pad_rows(W1.expand(k, d, h).contiguous())   # k <= E
    E, n = W1.shape[0], T * k
    perm = rng.permutation(n).astype(np.int32)
    offsets = np.full(E + 1, n, np.int32)
    offsets[0] = 0
    ws = moevie.Workspace(T, d, E, k, h)
    got = moevie.moevie_test_expert_hidden(x, dev(perm), dev(offsets), W1, k, ws)
    check_status(ws)
    rows = x[torch.from_numpy((perm // k).astype(np.int64)).cuda()].contiguous()
    ws1 = moevie.Workspace(n, d, 1, 1, h)
    one = moevie.moevie_pad_rows(W1[:1].contiguous())
    want = moevie.moevie_test_expert_hidden(rows, dev(np.arange(n, dtype=np.int32)), dev(np.array([0, n], np.int32)), one, 1, ws1)
    check_status(ws1)
    assert torch.equal(got, want)
