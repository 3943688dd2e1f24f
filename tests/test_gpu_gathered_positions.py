"""The tcgen05 kernels with gathered P rows (positions per token, lengths that no tile of sequences fits) and
the dispatch limits around them: ragged last tiles, one and two coordinate groups, with and without E rows,
positions and ids outside their tables."""

import numpy as np
import pytest
import torch

from oracle import ssn_oracle as oracle
from paper_2607_13332_b200 import binding as B
from paper_2607_13332_b200 import synth
from tests.harness import Codec, assert_close, f64, guards_intact, host64, padded, to_device

pytestmark = pytest.mark.gpu
DT = synth.BF16


@pytest.mark.parametrize("n,d,k,explicit", [
    (2369, 512, 40, True), (10007, 640, 8, True), (4999, 1024, 64, False), (19001, 512, 16, True),
    (515, 512, 72, True), (10007, 512, 128, False), (600, 768, 104, True)])
@pytest.mark.parametrize("tables", ["EP", "P"])
def test_gathered_positions(n, d, k, explicit, tables):
    wl = synth.Workload("gathered", d, k, 300, 1, n, DT)
    t = synth.codec_inputs(wl, seed=n + k, noise_std=0.05)
    E0, P0, rng = (t["E"] if "E" in tables else None), t["P"][:333], np.random.default_rng(n)
    seq = 333                                   # whole table, no multiple of 16
    pos, ids = rng.integers(0, 333, n).astype(np.int32), t["ids"].copy()
    if explicit:
        pos[[0, n - 1]] = [333, -1]             # outside: no P row, and the status bit
        ids[3] = 300 if E0 is not None else ids[3]
    else:
        pos = oracle.token_positions(n, seq)
    codec = Codec(DT, to_device(t["U"], DT), to_device(E0, DT), to_device(P0, DT))
    dids, dpos = torch.from_numpy(ids).cuda(), torch.from_numpy(pos).cuda() if explicit else None
    Z, zbuf = padded(n, k, k + 8, DT)
    codec.compress(to_device(t["X"], DT), dids, seq_len=seq, pos=dpos, out=Z)
    fam, var = B.ssn_last_kernel()
    assert fam == B.SSN_KERNEL_UMMA_PROJECT and var & B.SSN_KVAR_P and not var & B.SSN_KVAR_ALT
    expect, flags = oracle.compress(f64(t["X"], DT), f64(t["U"], DT), f64(E0, DT), ids, f64(P0, DT), pos)
    assert_close(host64(Z, DT), expect, DT, "compress")
    assert guards_intact(Z, zbuf, DT) and codec.take_status() == flags
    Z0, _ = padded(n, k, -(-k // 8) * 8, DT, fill=to_device(t["Z0"], DT))
    out, buf = padded(n, d, d + 64, DT)
    codec.decompress(Z0, dids, seq_len=seq, pos=dpos, out=out)
    fam, var = B.ssn_last_kernel()
    assert fam == B.SSN_KERNEL_UMMA_EXPAND and var & B.SSN_KVAR_P and not var & B.SSN_KVAR_ALT
    expect, flags = oracle.decompress(f64(t["Z0"], DT), f64(t["U"], DT), f64(E0, DT), ids, f64(P0, DT), pos)
    assert_close(host64(out, DT), expect, DT, "decompress")
    assert guards_intact(out, buf, DT) and codec.take_status() == flags


def test_few_rows_and_wire_rows_keep_their_kernels():
    """Up to 16 tokens per SM a small basis stays on the few-rows kernels; fp32 words from gathered rows come
    from the split kernel, accurate to fp32 sums (1e-6: see test_gpu_split_kernels)."""
    n, d, k = 1500, 512, 40
    wl = synth.Workload("few", d, k, 100, 1, n, DT)
    t = synth.codec_inputs(wl, seed=1, noise_std=0.05)
    pos = np.random.default_rng(0).integers(0, 99, n).astype(np.int32)
    codec = Codec(DT, to_device(t["U"], DT), to_device(t["E"], DT), to_device(t["P"], DT))
    ids, dpos, X = torch.from_numpy(t["ids"]).cuda(), torch.from_numpy(pos).cuda(), to_device(t["X"], DT)
    expect, _ = oracle.compress(f64(t["X"], DT), f64(t["U"], DT), f64(t["E"], DT), t["ids"], f64(t["P"], DT), pos)
    Z = codec.compress(X, ids, pos=dpos)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_MMA_SYNC_DSPLIT
    assert_close(host64(Z, DT), expect, DT, "compress")
    wire = codec.compress_wire(X, ids, pos=dpos)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_PROJECT
    assert_close(wire.view(torch.float32).double().cpu().numpy(), expect, DT, "wire", tol=1e-6)


@pytest.mark.parametrize("n,d,k,project,expand", [
    (3000, 1024, 16, B.SSN_KERNEL_MMA_SYNC_DSPLIT, B.SSN_KERNEL_MMA_SYNC_DSPLIT),
    (3000, 4096, 8, B.SSN_KERNEL_MMA_SYNC_DSPLIT, B.SSN_KERNEL_UMMA_EXPAND),
    (4736, 256, 64, B.SSN_KERNEL_MMA_SYNC_DSPLIT, None), (4736, 1024, 40, B.SSN_KERNEL_UMMA_PROJECT, B.SSN_KERNEL_UMMA_EXPAND),
    (4737, 512, 16, B.SSN_KERNEL_UMMA_PROJECT, None)])
def test_small_ranks_of_mid_sized_calls_keep_the_mma_sync_kernels(n, d, k, project, expand):
    wl = synth.Workload("mid", d, k, 100, 1, n, DT)
    t = synth.codec_inputs(wl, seed=n + k, noise_std=0.05)
    pos = np.random.default_rng(0).integers(0, 200, n).astype(np.int32)
    codec = Codec(DT, to_device(t["U"], DT), to_device(t["E"], DT), to_device(t["P"][:200], DT))
    ids, dpos = torch.from_numpy(t["ids"]).cuda(), torch.from_numpy(pos).cuda()
    U, E, P = f64(t["U"], DT), f64(t["E"], DT), f64(t["P"][:200], DT)
    Z = codec.compress(to_device(t["X"], DT), ids, pos=dpos)
    assert B.ssn_last_kernel()[0] == project
    assert_close(host64(Z, DT), oracle.compress(f64(t["X"], DT), U, E, t["ids"], P, pos)[0], DT, "compress")
    X = codec.decompress(to_device(t["Z0"], DT), ids, pos=dpos)
    assert expand is None or B.ssn_last_kernel()[0] == expand
    assert_close(host64(X, DT), oracle.decompress(f64(t["Z0"], DT), U, E, t["ids"], P, pos)[0], DT, "decompress")
