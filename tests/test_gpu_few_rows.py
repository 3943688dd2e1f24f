"""Projections of 512 to 16 tokens per SM: with E and P, as rows or as prepared tables, they stay on the
tcgen05 kernel, whose products are exact; without them the few-rows kernel is as exact and has the shorter start."""

import numpy as np
import pytest
import torch

from oracle import ssn_oracle as oracle
from paper_2607_13332_b200 import binding as B
from paper_2607_13332_b200 import synth
from tests.harness import Codec, f64, host64, to_device

pytestmark = pytest.mark.gpu
DT = synth.BF16
# Share of elements that are not the nearest bf16 value: fp32 sums are off by some 2e-6 of an element at most
# (192 truncated additions), bf16 neighbours are 2^-8 apart, so about one element in a thousand; a residual rounded to
# bf16 moves every element by about half the distance to its neighbour and misses a third of them.
MISSES = 0.01


def _misses(got: torch.Tensor, exact: np.ndarray) -> float:
    return float((got.float().cpu() != torch.from_numpy(exact).to(torch.bfloat16).float()).float().mean())


@pytest.mark.parametrize("batch,seq", [(4, 128), (16, 128), (37, 64), (1, 2368)])
@pytest.mark.parametrize("d,k", [(1024, 40), (512, 16), (256, 64)])
def test_small_calls_keep_exact_products_and_prepared_tables(batch, seq, d, k):
    wl = synth.Workload("few", d, k, 300, batch, seq, DT)
    t = synth.codec_inputs(wl, seed=batch + d + k, noise_std=0.05)
    codec = Codec(DT, to_device(t["U"], DT), to_device(t["E"], DT), to_device(t["P"], DT))
    ids, X = torch.from_numpy(t["ids"]).cuda(), to_device(t["X"], DT)
    pos = oracle.token_positions(wl.n_tokens, seq)
    expect, _ = oracle.compress(f64(t["X"], DT), f64(t["U"], DT), f64(t["E"], DT), t["ids"], f64(t["P"], DT), pos)
    if seq % 128 == 0:      # else the P rows of a tile are not consecutive and the rows keep the mma.sync kernels
        Z = codec.compress(X, ids, seq_len=seq)
        fam, var = B.ssn_last_kernel()
        assert fam == B.SSN_KERNEL_UMMA_PROJECT and var & B.SSN_KVAR_E and var & B.SSN_KVAR_P
        assert _misses(Z, expect) <= MISSES
    codec.prepare_tables()
    Z = codec.compress(X, ids, seq_len=seq)
    fam, var = B.ssn_last_kernel()
    assert fam == B.SSN_KERNEL_UMMA_PROJECT and not var & (B.SSN_KVAR_E | B.SSN_KVAR_P)
    assert _misses(Z, expect) <= MISSES
    plain = Codec(DT, to_device(t["U"], DT))
    dZ = plain.grad_project(to_device(t["G"], DT))
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_MMA_SYNC_DSPLIT
    assert _misses(dZ, oracle.grad_project_coeff(f64(t["G"], DT), f64(t["U"], DT))) <= MISSES
    assert codec.take_status() == 0


def test_wide_bases_stay_on_tcgen05():
    for d, k, family in ((4096, 16, B.SSN_KERNEL_MMA_SYNC_DSPLIT), (1024, 64, B.SSN_KERNEL_UMMA_PROJECT),
                         (2048, 40, B.SSN_KERNEL_UMMA_PROJECT)):
        U = synth.to_storage(synth.subspace_basis(d, k, seed=k), DT)
        G = synth.to_storage(np.random.default_rng(d).standard_normal((777, d)), DT)
        dZ = Codec(DT, to_device(U, DT)).grad_project(to_device(G, DT))
        assert B.ssn_last_kernel()[0] == family
        assert _misses(dZ, oracle.grad_project_coeff(f64(G, DT), f64(U, DT))) <= MISSES
