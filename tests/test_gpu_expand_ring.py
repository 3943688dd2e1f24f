"""The rings of gathered rows whose stages both epilogue groups of the tcgen05 expansion read in turn (E alone, and
E and P above rank 64): every pass of a batch of many chunks per CTA must repeat the first bit for bit."""

import pytest
import torch

from oracle import ssn_oracle as oracle
from paper_2607_13332_b200 import binding as B
from paper_2607_13332_b200 import synth
from tests.harness import Codec, assert_close, f64, host64, to_device

pytestmark = pytest.mark.gpu
DT = synth.BF16


@pytest.mark.parametrize("d,k,tables,batch,seq", [
    (640, 40, "E", 1, 20011), (2048, 64, "E", 1, 9000), (640, 104, "EP", 32, 640), (2048, 72, "EP", 16, 512), (1152, 40, "EP", 32, 640)])
def test_passes_repeat_and_match_the_oracle(d, k, tables, batch, seq):
    wl = synth.Workload("ring", d, k, 3000, batch, seq, DT)
    t = synth.codec_inputs(wl, seed=d + k, noise_std=0.05)
    P0 = t["P"] if "P" in tables else None
    codec = Codec(DT, to_device(t["U"], DT), to_device(t["E"], DT), to_device(P0, DT))
    ids, Z = torch.from_numpy(t["ids"]).cuda(), to_device(t["Z0"], DT)
    first = codec.decompress(Z, ids, seq_len=seq)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_UMMA_EXPAND
    expect, _ = oracle.decompress(f64(t["Z0"], DT), f64(t["U"], DT), f64(t["E"], DT), t["ids"], f64(P0, DT),
                                  oracle.token_positions(wl.n_tokens, seq))
    assert_close(host64(first, DT), expect, DT, "decompress")
    rows = torch.randperm(3000, device="cuda").to(torch.int32)
    for _ in range(20):                       # other rows in between, so that a stale stage would show
        codec.decompress(Z, rows[ids.long()], seq_len=seq)
        assert torch.equal(codec.decompress(Z, ids, seq_len=seq), first)
    assert codec.take_status() == 0
