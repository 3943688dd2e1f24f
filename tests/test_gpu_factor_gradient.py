"""The contraction over tokens behind the factor gradient: few and many blocks of columns, token counts that leave
one CTA, a few or sixteen per block, ranks whose rows take 16 bytes at a time and ranks whose rows do not."""

import numpy as np
import pytest
import torch

from paper_2607_13332_b200 import binding as B
from paper_2607_13332_b200 import synth
from paper_2607_13332_b200.runner import padded_columns
from tests.harness import Codec, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(512, 128), (1300, 130), (4096, 136), (520, 4096), (6443, 2048), (2624, 19000)])
@pytest.mark.parametrize("k", [8, 40, 51, 100])
def test_factor_gradient(n, m, k):
    d, dt = 128, synth.BF16
    g = torch.Generator(device="cuda").manual_seed(n + m + k)
    U = padded_columns(to_device(synth.to_storage(synth.subspace_basis(d, k, seed=k), dt), dt))
    H = padded_columns(torch.randn(n, m, device="cuda", generator=g).bfloat16())
    dY = torch.randn(n, d, device="cuda", generator=g).bfloat16()
    codec = Codec(dt, U)
    got = codec.reparam_grad_factor(H, dY)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_UMMA_TOKENS
    C = (dY.double() @ U.double()).bfloat16().double()          # the coordinates as they are stored in between
    expect = H.double().T @ C
    # fp32 sums of up to 6443 products, at most 80 truncated additions in a row (5e-7); one coordinate in a
    # thousand rounds to the other bf16 neighbour and moves the sums by 2^-8 / sqrt(1000 n)
    assert float((got.double() - expect).norm() / expect.norm()) <= 2e-4
    again = [codec.reparam_grad_factor(H, dY) for _ in range(3)]
    assert all(float((x - got).abs().max()) <= 2e-6 * np.sqrt(n) * float(C.std()) * 4 for x in again)
    assert codec.take_status() == 0
