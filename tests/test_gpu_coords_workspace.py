"""Project-then-expand of rows the fused kernel does not take (fp32 storage, operands off the 16-byte grid), through
fp32 coordinates in scratch: edges of the 128-row tiles and 128-column chunks, both rank groups, with and without the
coordinates as an output, and the general kernel where there is no scratch."""

import numpy as np
import pytest
import torch

from oracle import ssn_oracle as oracle
from paper_2607_13332_b200 import binding as B
from paper_2607_13332_b200 import synth
from tests.harness import Codec, assert_close, f64, guards_intact, host64, padded, to_device

pytestmark = pytest.mark.gpu

SPLIT = (B.SSN_KERNEL_SPLIT_PROJECT, B.SSN_KERNEL_SPLIT_EXPAND)


def _rand(rng, shape, dt, std=1.0):
    return synth.to_storage(rng.standard_normal(shape) * std, dt)


@pytest.mark.parametrize("dt", [synth.F32, synth.BF16])
@pytest.mark.parametrize("d,k,rows", [(130, 7, (300,)), (130, 7, (5000,)), (520, 7, (1, 127, 300)), (256, 51, (128, 129)), (384, 99, (700,)), (2048, 128, (513, 64))])
@pytest.mark.parametrize("scratch", [True, False])
def test_reprojection_of_rows(d, k, rows, dt, scratch):
    rng = np.random.default_rng(d + k)
    U0 = synth.to_storage(np.linalg.qr(rng.standard_normal((d, k)))[0], dt)
    W0 = [_rand(rng, (r, d), dt, 0.02) for r in rows]
    U, _ = padded(d, k, k + 1, dt, fill=to_device(U0, dt))       # off the 16-byte grid
    pairs = [padded(r, d, d + 3, dt, fill=to_device(w, dt)) for r, w in zip(rows, W0)]
    codec = Codec(dt, U)
    short = torch.empty(16, dtype=torch.uint8, device="cuda")    # too small to be of use
    codec.weight_reproject_list([w for w, _ in pairs], "right", workspace=None if scratch else short)
    # narrow rows, and calls without scratch, are the general kernel's
    assert (B.ssn_last_kernel()[0] in SPLIT) == (scratch and (d, rows) != (130, (300,)))
    for (w, buf), w0 in zip(pairs, W0):
        assert_close(host64(w, dt), oracle.weight_reproject(f64(w0, dt), f64(U0, dt), "right"), dt, "reproject")
        assert guards_intact(w, buf, dt)
    assert codec.take_status() == 0


@pytest.mark.parametrize("dt", [synth.F32, synth.BF16])
@pytest.mark.parametrize("n,m,d,k", [(1, 1000, 130, 5), (129, 320, 256, 51), (700, 130, 1100, 100), (3000, 512, 640, 17)])
@pytest.mark.parametrize("coords", [False, True])
def test_reparameterised_projection(n, m, d, k, dt, coords):
    rng = np.random.default_rng(n + m)
    H0, Zw0 = _rand(rng, (n, m), dt), _rand(rng, (m, k), dt, 0.02)
    U0 = synth.to_storage(np.linalg.qr(rng.standard_normal((d, k)))[0], dt)
    Zw, _ = padded(m, k, k + 1, dt, fill=to_device(Zw0, dt))
    out, buf = padded(n, d, d + 1, dt)
    C, cbuf = padded(n, k, k + 1, dt) if coords else (None, None)
    codec = Codec(dt, to_device(U0, dt))
    codec.reparam_project(to_device(H0, dt), Zw, out=out, coords=C)
    # bf16 coordinates as an output are the general kernel's
    assert (B.ssn_last_kernel()[0] in SPLIT) == (dt == synth.F32 or not coords)
    H, Z, U = f64(H0, dt), f64(Zw0, dt), f64(U0, dt)
    assert_close(host64(out, dt), oracle.reparam_project(H, Z, U), dt, "Y")
    assert guards_intact(out, buf, dt)
    if coords:
        assert_close(host64(C, dt), H @ Z, dt, "coordinates")
        assert guards_intact(C, cbuf, dt)
    assert codec.take_status() == 0


def test_a_workspace_given_to_a_right_list_is_left_alone():
    """Two such calls on two streams may be handed the same one; their weights would come out wrong if either wrote it."""
    d, k = 512, 40
    rng = np.random.default_rng(3)
    U0 = np.linalg.qr(rng.standard_normal((d, k)))[0].astype(np.float32)
    codec = Codec(synth.F32, to_device(U0, synth.F32))
    W0 = _rand(rng, (300, d), synth.F32, 0.02)
    given = torch.full((B.ssn_coords_workspace_bytes(codec.c, 300),), 0xA5, dtype=torch.uint8, device="cuda")
    weights = [to_device(W0, synth.F32) for _ in range(2)]
    codec.weight_reproject_list(weights[:1], "right", workspace=given)
    B.ssn_weight_reproject_list(codec.c, [weights[1].data_ptr()], [300], [d], B.SSN_SIDE_RIGHT, given.data_ptr(), given.numel(),
                                torch.cuda.current_stream().cuda_stream)
    assert bool((given == 0xA5).all())
    for w in weights:
        assert_close(host64(w, synth.F32), oracle.weight_reproject(f64(W0, synth.F32), f64(U0, synth.F32), "right"), synth.F32, "reproject")


def _reparam(seed, n=200, m=640, d=512, k=24):
    rng = np.random.default_rng(seed)
    H0, Zw0 = _rand(rng, (n, m), synth.F32), _rand(rng, (m, k), synth.F32, 0.02)
    U0 = np.linalg.qr(rng.standard_normal((d, k)))[0].astype(np.float32)
    expect = oracle.reparam_project(f64(H0, synth.F32), f64(Zw0, synth.F32), f64(U0, synth.F32))
    return Codec(synth.F32, to_device(U0, synth.F32)), to_device(H0, synth.F32), to_device(Zw0, synth.F32), expect


def test_requested_coordinates_need_no_scratch():
    codec, H, Zw, expect = _reparam(7)
    (n, m), k, d = H.shape, codec.k, codec.d
    Y, C = torch.empty((n, d), device="cuda"), torch.empty((n, k), device="cuda")
    B.ssn_reparam_project(codec.c, H.data_ptr(), m, m, Zw.data_ptr(), k, n, Y.data_ptr(), d, C.data_ptr(), k,
                          torch.cuda.current_stream().cuda_stream)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_EXPAND
    assert_close(Y.double().cpu().numpy(), expect, synth.F32, "Y")
    assert_close(C.double().cpu().numpy(), (H.double() @ Zw.double()).cpu().numpy(), synth.F32, "coordinates")


# calls on the 16-byte grid, but with fewer rows or other widths than the fused kernel takes
@pytest.mark.parametrize("n,m,d", [(300, 1024, 512), (700, 1024, 520), (700, 1000, 512), (511, 2048, 1024)])
@pytest.mark.parametrize("k", [8, 56])
def test_aligned_calls_the_fused_kernel_refuses(n, m, d, k):
    dt = synth.BF16
    rng = np.random.default_rng(n + m)
    H0, Zw0 = _rand(rng, (n, m), dt), _rand(rng, (m, k), dt, 0.02)
    U0 = synth.to_storage(np.linalg.qr(rng.standard_normal((d, k)))[0], dt)
    codec = Codec(dt, to_device(U0, dt))
    out = codec.reparam_project(to_device(H0, dt), to_device(Zw0, dt))
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_EXPAND
    assert_close(host64(out, dt), oracle.reparam_project(f64(H0, dt), f64(Zw0, dt), f64(U0, dt)), dt, "Y")


def test_aligned_weights_the_fused_kernel_refuses():
    d, k, dt = 1000, 40, synth.BF16
    rng = np.random.default_rng(5)
    U0 = synth.to_storage(np.linalg.qr(rng.standard_normal((d, k)))[0], dt)
    W0 = _rand(rng, (600, d), dt, 0.02)
    codec = Codec(dt, to_device(U0, dt))
    for call in (codec.weight_reproject, codec.weight_reproject_list):
        W = to_device(W0, dt)
        call([W], "right")
        assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_EXPAND
        assert_close(host64(W, dt), oracle.weight_reproject(f64(W0, dt), f64(U0, dt), "right"), dt, "reproject")


def test_no_memory_for_scratch(monkeypatch):
    codec, H, Zw, expect = _reparam(8)
    out = torch.empty((H.shape[0], codec.d), device="cuda")

    def full(*args, **kwargs):
        raise torch.OutOfMemoryError("no memory left")
    with monkeypatch.context() as m:
        m.setattr(torch, "empty", full)
        codec.reparam_project(H, Zw, out=out)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_GENERIC
    assert_close(out.double().cpu().numpy(), expect, synth.F32, "Y")
