"""Projection of bf16 rows as they are, with a basis at any address and pitch: rows of U that start on and between 4-byte
words, ranks on both sides of a lane's pair and of the 32- and 64-coordinate kernels, widths that end inside a stage, one
tile to several CTAs and several tiles to one; NaN around every operand, and infinite and NaN rows."""

import numpy as np
import pytest
import torch

from paper_2607_13332_b200 import binding as B
from paper_2607_13332_b200 import synth
from tests.harness import Codec, assert_close

pytestmark = pytest.mark.gpu

# fp32 words of exact products, up to 4096 of them added with compensation: the rounding of the result, 6e-8, and a few 2^-24
# of the partial sums, which are no larger than the rms at these inputs
WORD_TOL = 1e-6


def _rand(shape, seed, std=1.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(shape, device="cuda", generator=g) * std).bfloat16()


def _inside_nan(t, pitch, offset):
    """t at `offset` elements into a buffer of NaN, rows `pitch` apart."""
    rows, cols = t.shape
    buf = torch.full((offset + rows * pitch + 8,), float("nan"), dtype=t.dtype, device="cuda")
    view = torch.as_strided(buf, (rows, cols), (pitch, 1), offset)
    view.copy_(t)
    return view


def _variant():
    family, variant = B.ssn_last_kernel()
    assert family == B.SSN_KERNEL_SPLIT_PROJECT
    return variant


# up to 32 coordinates rows of more than one stage, or many; above that only wide rows, or many
NARROW = [(n, d, k) for n, d in [(1, 72), (127, 72), (129, 200), (700, 1000), (3000, 4096), (19100, 136), (30001, 24)] for k in (1, 2, 31, 32)]
WIDE = ([(n, d, k) for n, d in [(5000, 2056), (19100, 1032)] for k in (33, 51, 63, 64, 65, 99, 127, 128)]
        + [(3000, 4096, k) for k in (51, 64, 127)] + [(1, 2056, k) for k in (33, 64)])


@pytest.mark.parametrize("n,d,k", [c for c in NARROW if c[2] <= c[1]] + WIDE)
@pytest.mark.parametrize("excess,offset", [(0, 0), (1, 1), (2, 3), (3, 8)])
def test_any_basis(n, d, k, excess, offset):
    if (k + excess) % 8 == 0 and offset % 8 == 0:
        excess += 2   # an aligned basis belongs to the TMA kernels
    X = _inside_nan(_rand((n, d), n), (d + 15) // 8 * 8, 64)
    U = _inside_nan(_rand((d, k), k, d ** -0.5), k + excess, offset)
    codec = Codec(synth.BF16, U)
    expect = (X.double() @ U.double()).cpu().numpy()
    words = torch.full((n, k + 2), -1, dtype=torch.int32, device="cuda")
    codec.grad_project_wire(X, out=words.view(torch.float32)[:, :k])
    variant = _variant()
    assert variant & B.SSN_KVAR_PLAIN and bool(variant & B.SSN_KVAR_WIDE) == (k > 64)
    # 150 tiles and more, or 80 halves of tiles: single CTAs; fewer, of two stages or more: several CTAs to a tile
    assert bool(variant & B.SSN_KVAR_ALT) == (n < 5000 or n == 5000 and k <= 64)
    assert_close(words.view(torch.float32)[:, :k].double().cpu().numpy(), expect, synth.F32, "words", tol=WORD_TOL)
    assert (words[:, k:] == -1).all()
    Z = codec.grad_project(X)
    assert _variant() & B.SSN_KVAR_PLAIN
    assert_close(Z.double().cpu().numpy(), expect, synth.BF16, "rows")
    ids = torch.arange(n, dtype=torch.int32, device="cuda")
    wire = codec.compress_wire(X, ids, with_ids=True)
    assert _variant() & B.SSN_KVAR_PLAIN
    assert torch.equal(wire[:, k], ids) and torch.equal(wire[:, :k], words[:, :k])
    assert codec.take_status() == 0


# clusters and single CTAs of both kernels, for few and for many coordinates
@pytest.mark.parametrize("n,d,k,plain,cluster", [(300, 256, 27, True, True), (20000, 256, 27, True, False), (300, 2048, 51, True, True),
                                                 (20000, 1032, 64, True, False), (300, 256, 51, False, True), (20000, 256, 51, False, False),
                                                 (300, 64, 27, False, False)])
def test_bad_rows(n, d, k, plain, cluster):
    X, U = _rand((n, d), 1), _inside_nan(_rand((d, k), 2, d ** -0.5), k + 1 + k % 2, 0)
    X[0, 5], X[129, 9], X[130, 9] = float("inf"), -float("inf"), float("nan")
    X[20] *= 1e36
    X[21] = 3e38                                  # sums out of the range of fp32, at the end or on the way
    codec = Codec(synth.BF16, U)
    got = codec.grad_project_wire(X).double().cpu().numpy()
    variant = _variant()
    assert bool(variant & B.SSN_KVAR_PLAIN) == plain and bool(variant & B.SSN_KVAR_ALT) == cluster
    expect = (X.double() @ U.double()).float().double().cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(expect))
    assert np.array_equal(np.isinf(got), np.isinf(expect))
    rows = np.isfinite(expect).all(axis=1)
    scale = np.abs(expect[rows]).max(axis=1, keepdims=True)
    assert (np.abs(got[rows] - expect[rows]) <= 1e-5 * scale).all()
    finite = np.isfinite(expect[21])
    assert np.allclose(got[21, finite], expect[21, finite], rtol=1e-5)
    # a bad value of the basis stays in its column
    U[7, 3] = float("nan")
    got = Codec(synth.BF16, U).grad_project_wire(X[200:]).cpu().numpy()
    assert np.isnan(got[:, 3]).all() and np.isfinite(np.delete(got, 3, axis=1)).all()


# 2-norm of the error against 64-bit sums.  Few terms per CTA (up to 320 columns, or wider rows dealt to a cluster): added with
# compensation one by one the four accumulators of a stage give 4.0e-8 to 4.93e-8, in plain fp32 5.2e-8 to 6.0e-8.  Rows of the
# subspace, two long slices: 3.0e-8 with the compensations of both, 3.8e-8 with their rounded sums.
@pytest.mark.parametrize("n,d,k,coherent,bound", [(20000, 192, 32, 0, 5.05e-8), (20000, 256, 19, 0, 5.05e-8), (20000, 320, 32, 0, 5.05e-8),
                                                  (3000, 1024, 19, 0, 5.05e-8), (9000, 640, 32, 0, 5.05e-8), (700, 2048, 51, 0, 5.05e-8),
                                                  (3000, 5120, 99, 1, 3.4e-8)])
def test_words_of_few_terms(n, d, k, coherent, bound):
    X, U = _rand((n, d), n), _rand((d, k), k, d ** -0.5)
    if coherent:
        X = (_rand((n, k), 3, 3.0).float() @ U.float().T + 0.3 * X.float()).bfloat16()
    got = Codec(synth.BF16, _inside_nan(U, k + 1 + k % 2, 0)).grad_project_wire(X).double()
    assert _variant() & B.SSN_KVAR_PLAIN
    expect = X.double() @ U.double()
    assert (got - expect).norm() <= bound * expect.norm()
