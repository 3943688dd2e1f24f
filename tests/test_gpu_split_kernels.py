"""The split-operand tcgen05 kernels (fp32 storage, and the bf16 calls TMA cannot fetch) at the sizes
where they can go wrong: edges of the 128-token tiles, the 64-column stages and the 128-column chunks,
one and several CTAs per tile, every rank variant, leading dimensions off the 16-byte grid, positions
per token; and rows whose magnitudes the three-part split does not hold."""

import numpy as np
import pytest
import torch

from oracle import ssn_oracle as oracle
from paper_2607_13332_b200 import binding as B
from paper_2607_13332_b200 import synth
from tests.harness import Codec, assert_close, f64, guards_intact, host64, padded, to_device

pytestmark = pytest.mark.gpu

# fp32 sums of at most 2176 products of size ~1/sqrt(d): 64-column chains of fp32 additions err by a few
# 2^-24 of the partial sums, 1e-6 of the rms at the outer tail over all elements of a result
F32_SUM_TOL = 1e-6

CASES = [   # n, d, k, leading dimension excess (elements)
    (1, 64, 1, 1), (127, 65, 7, 0), (128, 127, 32, 1), (129, 128, 33, 0), (300, 192, 64, 3), (513, 130, 65, 1),
    (2000, 2176, 40, 0), (2000, 1088, 128, 1), (10007, 256, 51, 0), (19100, 136, 9, 1), (40000, 72, 17, 0),
]


def _inputs(n, d, k, dt, seed):
    wl = synth.Workload("split", d, k, 97, 1, n, dt)
    return synth.codec_inputs(wl, seed=seed, noise_std=0.05)


def _strided(t, dt, excess):
    t = to_device(t, dt)
    view, _ = padded(t.shape[0], t.shape[1], t.shape[1] + excess, dt, fill=t)
    return view


@pytest.mark.parametrize("n,d,k,excess", CASES)
@pytest.mark.parametrize("dt", [synth.F32, synth.BF16])
@pytest.mark.parametrize("tables", ["EP", "E", "none"])
def test_split_kernels_match_the_oracle(n, d, k, excess, dt, tables):
    if dt == synth.BF16 and excess == 0 and k % 8 == 0 and d % 8 == 0:
        excess = 1   # an aligned bf16 call belongs to the TMA kernels
    rng = np.random.default_rng(n + d)
    t = _inputs(n, d, k, dt, seed=n + k)
    E0, P0 = (t["E"] if "E" in tables else None), (t["P"][:50] if "P" in tables else None)
    pos = rng.integers(0, min(50, n), n).astype(np.int32)
    dev = {x: _strided(t[x], dt, excess) for x in ("X", "G", "U", "Z0")}
    codec = Codec(dt, dev["U"], None if E0 is None else _strided(E0, dt, excess), None if P0 is None else _strided(P0, dt, excess))
    ids, dpos = torch.from_numpy(t["ids"]).cuda(), torch.from_numpy(pos).cuda()
    f = {x: f64(t[x], dt) for x in ("X", "G", "U", "Z0")}
    E, P = f64(E0, dt), f64(P0, dt)

    Z, buf = padded(n, k, k + excess, dt)
    codec.compress(dev["X"], ids, pos=dpos, out=Z)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_PROJECT
    expect, _ = oracle.compress(f["X"], f["U"], E, t["ids"], P, pos)
    assert_close(host64(Z, dt), expect, dt, "compress", tol=F32_SUM_TOL if dt == synth.F32 else None)
    assert guards_intact(Z, buf, dt)

    # a residual addend beside the tables, fp32 words out with the token id
    wire = codec.compress_sum(dev["X"], dev["G"], ids, pos=dpos, wire=True, with_ids=True)
    expect, _ = oracle.compress_sum(f["X"], f["G"], f["U"], E, t["ids"], P, pos)
    coords, got_ids = oracle.wire_unpack(wire.cpu().numpy(), k, True)
    if tables != "none" or excess or dt == synth.F32:
        assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_PROJECT
        assert_close(coords, expect, dt, "compress_sum wire", tol=F32_SUM_TOL)
    assert np.array_equal(got_ids, t["ids"])

    out, buf = padded(n, d, d + excess, dt)
    codec.decompress(dev["Z0"], ids, pos=dpos, out=out)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_EXPAND
    expect, _ = oracle.decompress(f["Z0"], f["U"], E, t["ids"], P, pos)
    assert_close(host64(out, dt), expect, dt, "decompress", tol=F32_SUM_TOL if dt == synth.F32 else None)
    assert guards_intact(out, buf, dt)

    Xw = codec.decompress_wire(wire, pos=dpos, with_ids=True, use_workspace=False)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_EXPAND
    expect, _ = oracle.decompress(coords, f["U"], E, t["ids"], P, pos)
    assert_close(host64(Xw, dt), expect, dt, "decompress_wire", tol=F32_SUM_TOL if dt == synth.F32 else None)
    assert codec.take_status() == 0


def _same_as_plain_sums(got, expect, what):
    """Infinities and NaN where plain sums have them; each other row within the fp32 tolerance of its own scale."""
    assert np.array_equal(np.isnan(got), np.isnan(expect)), what
    inf = np.isinf(expect)
    assert np.array_equal(np.isinf(got), inf) and np.array_equal(np.sign(got[inf]), np.sign(expect[inf])), what
    for r in range(expect.shape[0]):
        if np.isfinite(expect[r]).all():
            scale = max(np.abs(expect[r]).max(), 1e-300)
            assert np.abs(got[r] - expect[r]).max() <= 1e-5 * scale, (what, r)


@pytest.mark.parametrize("n,d,k", [(300, 256, 40), (19100, 128, 16)])
def test_rows_the_split_does_not_hold(n, d, k):
    """Infinite, NaN, enormous and tiny rows (and one row of zeros) give what plain fp32 sums give."""
    dt = synth.F32
    t = _inputs(n, d, k, dt, seed=3)
    t["X"][0, 5], t["X"][7, 9], t["X"][8, 9] = np.inf, -np.inf, np.nan
    t["X"][20] *= 1e36
    t["X"][130] *= 1e-30
    t["X"][131] = 0
    t["Z0"][0, 3], t["Z0"][9, 0] = np.inf, np.nan
    t["Z0"][21] *= 1e36
    t["Z0"][130] *= 1e-30
    codec = Codec(dt, to_device(t["U"], dt))
    f = {x: f64(t[x], dt) for x in ("X", "U", "Z0")}
    with np.errstate(invalid="ignore"):
        _same_as_plain_sums(host64(codec.grad_project(to_device(t["X"], dt)), dt), f["X"] @ f["U"], "projection")
        _same_as_plain_sums(host64(codec.decompress(to_device(t["Z0"], dt)), dt), f["Z0"] @ f["U"].T, "expansion")
        # an infinity in the basis concerns every row
        t["U"][3, 1] = np.inf
        U = f64(t["U"], dt)
        codec = Codec(dt, to_device(t["U"], dt))
        finite = _inputs(n, d, k, dt, seed=4)
        X, Z = f64(finite["X"], dt), f64(finite["Z0"], dt)
        _same_as_plain_sums(host64(codec.grad_project(to_device(finite["X"], dt)), dt), X @ U, "projection, U")
        _same_as_plain_sums(host64(codec.decompress(to_device(finite["Z0"], dt)), dt), Z @ U.T, "expansion, U")
    assert codec.take_status() == 0


@pytest.mark.parametrize("k", [72, 100, 127])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_a_bad_basis_value_stays_in_its_column(k, bad):
    """Above rank 64 a stage of U serves both groups of 64 coordinates, of one chunk of columns after the other:
    an infinity or NaN in row r of U belongs to output column r and to no column of another chunk."""
    n, d, dt = 4000, 1664, synth.BF16                   # 32 x 13 units, several per CTA
    t = _inputs(n, d, k, dt, seed=k)
    U = t["U"].copy()
    U[[5, 700, 1663], [40, 15, 63]] = synth.to_storage(np.array([bad], np.float64), dt)[0]
    codec = Codec(dt, _strided(U, dt, 3))
    finite = np.setdiff1d(np.arange(d), [5, 700, 1663])
    expect = f64(t["Z0"], dt) @ f64(t["U"], dt).T
    out = host64(codec.decompress(_strided(t["Z0"], dt, 3)), dt)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_EXPAND
    assert_close(out[:, finite], expect[:, finite], dt, "decompress")
    assert not np.isfinite(out[:, [5, 700, 1663]]).any()
    wire = torch.from_numpy(f64(t["Z0"], dt).astype(np.float32)).cuda().view(torch.int32)
    out = host64(codec.decompress_wire(wire, use_workspace=False), dt)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_EXPAND
    assert_close(out[:, finite], expect[:, finite], dt, "decompress_wire")
    assert not np.isfinite(out[:, [5, 700, 1663]]).any()


def _close_per_column(got, expect, what):
    scale = np.abs(expect).max(axis=0)
    assert (np.abs(got - expect).max(axis=0) <= 1e-5 * scale).all(), what


@pytest.mark.parametrize("n,d,k", [(300, 256, 40), (19100, 130, 17), (700, 1100, 72)])
@pytest.mark.parametrize("scale", [1e-33, 1e-37, 1e13])
def test_columns_and_rows_of_a_basis_the_split_does_not_hold(n, d, k, scale):
    """A column of U (projection) or a row of it (expansion) that is tiny or enormous as a whole keeps the precision of
    fp32 against its own size; tiny values beside ordinary ones are no reason to compute anything again."""
    dt = synth.F32
    t = _inputs(n, d, k, dt, seed=5)
    X, Z = f64(t["X"], dt), f64(t["Z0"], dt)
    col, row = t["U"].copy(), t["U"].copy()
    col[:, 3] *= np.float32(scale)
    col[5, 2] = 1e-36
    row[7] *= np.float32(scale)
    row[9, 1] = 1e-36
    dev = Codec(dt, to_device(col, dt))
    _close_per_column(host64(dev.grad_project(to_device(t["X"], dt)), dt), X @ f64(col, dt), "projection")
    dev = Codec(dt, to_device(row, dt))
    _close_per_column(host64(dev.decompress(to_device(t["Z0"], dt)), dt), Z @ f64(row, dt).T, "expansion")


@pytest.mark.parametrize("n,d", [(300, 256), (19100, 128)])     # one tile to a cluster of CTAs; a CTA with several tiles
@pytest.mark.parametrize("dt", [synth.F32, synth.BF16])
@pytest.mark.parametrize("addend", [False, True])
def test_bad_rows_beside_tables_and_addends(n, d, dt, addend):
    """Rows the split does not hold, beside E and P rows and a residual addend and as fp32 wire words; a row whose first
    columns alone are tiny; every other row is what it is without them."""
    k, ld = 40, 1
    t = _inputs(n, d, k, dt, seed=11)
    rng = np.random.default_rng(1)
    pos = rng.integers(0, 50, n).astype(np.int32)
    X, R = f64(t["X"], dt), f64(t["G"], dt)
    X[0, 5], X[129, 9], X[130, 9] = np.inf, -np.inf, np.nan
    X[20] *= 1e36
    X[131, :32] = 1e-30
    Xs, Rs = synth.to_storage(X, dt), synth.to_storage(R, dt)
    X, R, E, P, U = f64(Xs, dt), f64(Rs, dt), f64(t["E"], dt), f64(t["P"][:50], dt), f64(t["U"], dt)
    codec = Codec(dt, _strided(t["U"], dt, ld), _strided(t["E"], dt, ld), _strided(t["P"][:50], dt, ld))
    ids, dpos = torch.from_numpy(t["ids"]).cuda(), torch.from_numpy(pos).cuda()
    with np.errstate(invalid="ignore"):
        if addend:
            wire = codec.compress_sum(_strided(Xs, dt, ld), _strided(Rs, dt, ld), ids, pos=dpos, wire=True)
            expect, _ = oracle.compress_sum(X, R, U, E, t["ids"], P, pos)
        else:
            wire = codec.compress_wire(_strided(Xs, dt, ld), ids, pos=dpos)
            expect, _ = oracle.compress(X, U, E, t["ids"], P, pos)
        assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_PROJECT
        got = wire.view(torch.float32).double().cpu().numpy()
        _same_as_plain_sums(got, expect, "projection")
        # fp32 coordinates into bf16 rows: tiny, enormous and infinite ones
        Z = f64(t["Z0"], dt).astype(np.float32)
        Z[3, 1], Z[4] = np.inf, Z[4] * np.float32(1e-30)
        Z[5] *= np.float32(1e36)
        out = host64(codec.decompress_wire(torch.from_numpy(Z).cuda().view(torch.int32), ids, pos=dpos, use_workspace=False), dt)
        assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_EXPAND
        expect, _ = oracle.decompress(Z.astype(np.float64), U, E, t["ids"], P, pos)
        rows = np.setdiff1d(np.arange(n), [3])
        ok = np.abs(out[rows] - expect[rows]).max(axis=1) <= (1e-5 if dt == synth.F32 else 1e-2) * np.abs(expect[rows]).max(axis=1)
        assert ok.all()
        assert not np.isfinite(out[3]).any()
    assert codec.take_status() == 0


@pytest.mark.parametrize("dt", [synth.F32, synth.BF16])
@pytest.mark.parametrize("n", [700, 4096, 20000])               # eight, a few and one CTA per tile
@pytest.mark.parametrize("d", [128, 256, 1024, 4096])
@pytest.mark.parametrize("k", [8, 40, 100])
def test_sums_as_accurate_as_plain_fmas(n, d, k, dt):
    """Error of fp32 coordinates against 64-bit sums, 2-norm over 2-norm.  The rounding of a result alone is 2.5e-8.  Plain
    FMAs over 32 lanes measure 4.0e-8 to 6.7e-8 on rows of the subspace (terms of one sign) and 4.8e-8 to 2.1e-7 on
    random ones; chains of truncated additions without compensation 6.4e-8 to 1.3e-7 and 5.3e-8 to 1.7e-7.  The
    bounds lie a tenth above this kernel's own 4.8e-8 to 6.1e-8 and 5.1e-8 to 6.9e-8."""
    g = torch.Generator(device="cuda").manual_seed(n + d + k)
    tdt = torch.float32 if dt == synth.F32 else torch.bfloat16
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)
    U = torch.zeros((d, k + 1), device="cuda", dtype=tdt)
    U[:, :k] = torch.linalg.qr(rnd(d, k))[0]
    U = U[:, :k]                                                # off the 16-byte grid
    E, ids = (0.1 * rnd(500, d)).to(tdt), torch.randint(0, 500, (n,), device="cuda", dtype=torch.int32, generator=g)
    rows, noise = rnd(n, k) @ U.float().T, rnd(n, d)

    def error(got, exact):
        return float((got.double() - exact).norm() / exact.norm())

    for name, x, bound in (("subspace", rows.to(tdt), 6.2e-8), ("random", noise.to(tdt), 7.5e-8)):
        exact = x.double() @ U.double()
        got = Codec(dt, U).grad_project_wire(x)
        assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_PROJECT
        assert error(got, exact) <= bound, name
    x = (rows + E[ids.long()].float() + 0.05 * noise).to(tdt)
    got = Codec(dt, U, E).compress_wire(x, ids).view(torch.float32)
    assert B.ssn_last_kernel()[0] == B.SSN_KERNEL_SPLIT_PROJECT
    assert error(got, (x.double() - E[ids.long()].double()) @ U.double()) <= 7.5e-8, "residual"
