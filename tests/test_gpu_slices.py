"""The sliced sweep (the default path of every product and sweep): sizes
around a slice of 32 rows, 16-bit and int32 columns, one to five interleaved
right-hand sides at 16- and 8-byte alignment, padding next to infinite
entries, and new values after a refactorisation."""
import numpy as np
import pytest

import oracle
import synth
from _helpers import maxabs_err, relerr

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP64_TOL = 1e-12


@pytest.fixture(scope="module")
def silu():
    import paper_2111_09512_gb300 as s
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s.build()
    return s


@pytest.fixture(scope="module")
def ctx(silu):
    return silu.Context(0, torch.cuda.current_stream())


def dev(a, shift=0):
    """A contiguous device copy whose address is 8 * shift bytes past a 256-byte boundary."""
    a = np.ascontiguousarray(a)
    buf = torch.empty(a.size + shift, dtype=torch.float64, device="cuda")
    t = buf[shift:].view(a.shape)
    t.copy_(torch.from_numpy(a))
    return t


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def far(n, reach):
    """Tridiagonal plus couplings `reach` rows away (diagonally dominant)."""
    i = np.arange(n)
    rows, cols = [i], [i]
    for d in (1, reach):
        rows += [i[d:], i[:-d]]
        cols += [i[:-d], i[d:]]
    r, c = np.concatenate(rows), np.concatenate(cols)
    order = np.lexsort((c, r))
    r, c = r[order], c[order]
    v = np.where(r == c, 5.0, -synth.uniform(5, 1, len(r), 0.1, 1.0))
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, r + 1, 1)
    return np.cumsum(rp), c.astype(np.int32), v


CASES = [
    ("1 row", lambda: synth.banded(1, 0, 1, seed=12)),
    ("31 rows", lambda: synth.banded(31, 5, 31, seed=11)),
    ("32 rows", lambda: synth.banded(32, 4, 12, seed=3)),
    ("33 rows", lambda: synth.banded(33, 3, 8, seed=10)),
    ("cutcell 37x29x23", lambda: synth.cutcell7(37, 29, 23, seed=1)),
    ("hex27 17x13x11", lambda: synth.hex27(17, 13, 11, seed=3)),
    ("columns 65534 apart", lambda: far(65600, 65534 // 2 - 16)),
    ("columns beyond 16 bits", lambda: far(66100, 66001)),
]


@pytest.mark.parametrize("shift", [0, 1], ids=["aligned", "odd"])
@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_sliced_products_and_sweeps_match_oracle(silu, ctx, case, shift):
    A = case[1]()
    n = len(A[0]) - 1
    M = silu.Matrix(ctx, *A)
    F = silu.ilu_setup(ctx, M, "ilu0")
    F.set_fused(1)
    F32 = silu.ilu_setup(ctx, M, "ilu0", prec=silu.FP32)
    F32.set_fused(1)
    S = oracle.row_scale(oracle.factor(A, "ilu0", 0.0, 0))
    for nrhs in (1, 2, 3, 4, 5):
        b, x0 = synth.rhs(n, nrhs, seed=21), synth.rhs(n, nrhs, seed=22) * 0.5
        r = dev(np.zeros((n, nrhs)), shift)
        M.residual(r, dev(x0, shift), dev(b, shift))
        assert maxabs_err(host(r), oracle.residual(A, x0, b)) < FP64_TOL, nrhs
        for mL, mU in [(3, 4), (1, 1), (2, 0)]:
            want = oracle.smooth(A, S, x0, b, mL, mU)
            for G, tol in ((F, FP64_TOL), (F32, 1e-5)):
                x = dev(x0, shift)
                silu.ilu_smooth(G, x, dev(b, shift), mL, mU)
                ctx.check()
                got = host(x)
                for k in range(nrhs):
                    assert relerr(got[:, k], want[:, k]) < tol, (nrhs, mL, mU, k)


@pytest.mark.parametrize("name,gen", [CASES[4], CASES[7]], ids=[CASES[4][0], CASES[7][0]])
def test_sliced_sweeps_give_the_tiled_sweeps_bits(silu, ctx, name, gen):
    """One lane sums a row in column order on slices as on tiles."""
    A = gen()
    n = len(A[0]) - 1
    b, x0 = synth.rhs(n, 1, seed=1), synth.rhs(n, 1, seed=2)
    for prec in (silu.FP64, silu.FP32):
        F = silu.ilu_setup(ctx, silu.Matrix(ctx, *A), "ilut", 1e-3, 10, prec=prec)
        out = []
        for variant in (0, 2):
            F.set_kernel(variant)
            x = dev(x0)
            silu.ilu_smooth(F, x, dev(b), 6, 5)
            out.append(host(x))
        assert np.array_equal(out[0], out[1])


def test_padding_reads_no_vector_entry(silu, ctx):
    """An infinite or NaN entry of x reaches only the rows that refer to it."""
    A = synth.cutcell7(21, 17, 13, seed=5)
    n = len(A[0]) - 1
    rp, ci, _ = A
    b, x = synth.rhs(n, 1, seed=3), synth.rhs(n, 1, seed=4)
    clean = oracle.residual(A, x, b)[:, 0]
    M = silu.Matrix(ctx, *A)
    for j, bad in ((0, np.inf), (n // 2, np.nan), (n - 1, -np.inf)):
        xb = x.copy()
        xb[j] = bad
        r = dev(np.zeros((n, 1)))
        M.residual(r, dev(xb), dev(b))
        got = host(r)[:, 0]
        hit = np.zeros(n, bool)
        for i in range(n):
            hit[i] = j in ci[rp[i]:rp[i + 1]]
        assert not np.isfinite(got[hit]).any() and relerr(got[~hit], clean[~hit]) < FP64_TOL


def test_refactor_renews_the_slices_of_the_matrix(silu, ctx):
    A, A2 = synth.cutcell7(19, 18, 17, seed=3), synth.cutcell7(19, 18, 17, seed=8)
    n = len(A[0]) - 1
    M = silu.Matrix(ctx, *A)
    F = silu.ilu_setup(ctx, M, "ilu0")
    silu.ilu_refactor(F, A2[2])
    b, x0 = synth.rhs(n, 1, seed=5), synth.rhs(n, 1, seed=6)
    S = oracle.row_scale(oracle.factor(A2, "ilu0", 0.0, 0))
    x = dev(x0)
    silu.ilu_smooth(F, x, dev(b), 4, 4)
    assert relerr(host(x), oracle.smooth(A2, S, x0, b, 4, 4)) < FP64_TOL
    r = dev(np.zeros((n, 1)))
    M.residual(r, dev(x0), dev(b))
    assert relerr(host(r), oracle.residual(A2, x0, b)) < FP64_TOL


# one, one and a bit, eight and a bit, sixteen and sixteen and a bit slices of 32 rows per SM of 152
SMALL = [pytest.param(size, gen, kind, id=f"{gen}-{kind}-{'x'.join(map(str, size))}")
         for size in ((12, 11, 13), (17, 16, 18), (34, 34, 34), (43, 43, 42), (43, 43, 44))
         for gen, kind in (("cutcell7", "ilu0"), ("cutcell7", "ilut"), ("hex27", "ilu0"))]


@pytest.mark.parametrize("size,gen,kind", SMALL)
def test_small_systems_match_the_lanes_per_row_kernel(silu, ctx, size, gen, kind):
    """Automatic choice (small sliced kernels or the fused launch) against the general kernel: sums of
    at most 28 terms of a scaled system, eight sweeps, so rounding of order 1e-14 (FP32 1e-5)."""
    A = getattr(synth, gen)(*size, seed=6)
    n = len(A[0]) - 1
    M = silu.Matrix(ctx, *A)
    for scale in (silu.SCALE_ROW, silu.SCALE_ROWCOL):
        for prec, tol in ((silu.FP64, FP64_TOL), (silu.FP32, 1e-5)):
            F = silu.ilu_setup(ctx, M, kind, 1e-3, 10, scale=scale, prec=prec)
            for nrhs in (1, 2, 3, 4):
                b, x0 = synth.rhs(n, nrhs, seed=7), synth.rhs(n, nrhs, seed=8)
                out = []
                for variant, fused in ((0, 0), (1, 1), (0, 2)):
                    F.set_kernel(variant)
                    F.set_fused(fused)
                    x = dev(x0)
                    silu.ilu_smooth(F, x, dev(b), 5, 4)
                    ctx.check()
                    out.append(host(x))
                assert max(relerr(out[0][:, k], out[1][:, k]) for k in range(nrhs)) < tol, (scale, prec, nrhs)
                if prec == silu.FP32 and nrhs in (2, 4):  # the fused launch's order of summation
                    assert np.array_equal(out[0], out[2]), (scale, nrhs)


@pytest.mark.parametrize("gen", [lambda: synth.hex27(46, 45, 44, seed=2), lambda: synth.hex27(262, 258, 5, seed=2)],
                         ids=["16-bit columns", "int32 columns"])
def test_long_rows_and_int32_columns_match_the_lanes_per_row_kernel(silu, ctx, gen):
    """Rows of up to 13 factor entries on both sides of the lines between slices and tiles."""
    A = gen()
    n = len(A[0]) - 1
    M = silu.Matrix(ctx, *A)
    for prec, tol in ((silu.FP64, FP64_TOL), (silu.FP32, 1e-5)):
        F = silu.ilu_setup(ctx, M, "ilu0", prec=prec)
        for nrhs in (1, 2, 3, 4):
            b, x0 = synth.rhs(n, nrhs, seed=9), synth.rhs(n, nrhs, seed=10)
            out = []
            for variant, fused in ((0, 0), (1, 1)):
                F.set_kernel(variant)
                F.set_fused(fused)
                x = dev(x0)
                silu.ilu_smooth(F, x, dev(b), 3, 4)
                ctx.check()
                out.append(host(x))
            assert max(relerr(out[0][:, k], out[1][:, k]) for k in range(nrhs)) < tol, (prec, nrhs)


def test_lanes_asked_for_are_used(silu, ctx):
    """silu_ilu_set_lanes shapes the sweeps of several columns of the automatic variant: the bits of variant 1, not
    those of the sliced sweeps (an eight-lane sum of up to 10 terms rounds differently in some row)."""
    A = synth.cutcell7(21, 19, 17, seed=2)
    n = len(A[0]) - 1
    for prec in (silu.FP64, silu.FP32):
        F = silu.ilu_setup(ctx, silu.Matrix(ctx, *A), "ilut", 1e-3, 10, prec=prec)
        F.set_fused(1)
        for nrhs in (2, 3, 4):
            b, x0 = synth.rhs(n, nrhs, seed=5), synth.rhs(n, nrhs, seed=6)
            out = {}
            for variant, lanes in ((0, 0), (0, 8), (1, 8)):
                F.set_kernel(variant)
                F.set_lanes(lanes, lanes, lanes)
                x = dev(x0)
                silu.ilu_smooth(F, x, dev(b), 4, 4)
                out[variant, lanes] = host(x)[:, :nrhs // 2 * 2]  # a third column goes by itself, on tiles or slices
            assert np.array_equal(out[0, 8], out[1, 8]), (prec, nrhs)
            if prec == silu.FP64:
                assert not np.array_equal(out[0, 8], out[0, 0]), nrhs


def test_a_shape_for_one_column_leaves_several_columns_alone(silu, ctx):
    """silu_mat_set_shape and its autotuner time one column; blocks of columns keep the sliced kernel's bits."""
    A = synth.cutcell7(21, 19, 17, seed=2)
    n = len(A[0]) - 1
    M = silu.Matrix(ctx, *A)
    F = silu.ilu_setup(ctx, M, "ilu0")
    F.set_fused(1)
    for nrhs in (2, 3, 4, 5):
        b, x0 = synth.rhs(n, nrhs, seed=5), synth.rhs(n, nrhs, seed=6)
        out = []
        for shape in ((0, 0, 0), (4, 1, 16), (1, 2, 16)):
            M.set_shape(*shape)
            r, x = dev(np.zeros((n, nrhs))), dev(x0)
            M.residual(r, x, dev(b))
            silu.ilu_smooth(F, x, dev(b), 3, 3)
            out.append((host(r), host(x)))
        assert all(np.array_equal(p, q) for o in out[1:] for p, q in zip(out[0], o)), nrhs


# FP32 factors of at least 64 slices of 32 rows per SM: units of four, two and one slices, several units per warp
# (stages are used again), the last unit and the last slice not full
RING = [("ilu0", "cutcell7", (111, 109, 107), 0, 4), ("iluk", "cutcell7", (91, 89, 85), 1, 2),
        ("ilu0", "hex27", (80, 71, 59), 0, 1)]


@pytest.mark.parametrize("kind,gen,size,fill,unit", RING, ids=["4 slices", "2 slices", "1 slice"])
def test_large_fp32_sweeps_through_the_ring(silu, ctx, kind, gen, size, fill, unit):
    """One lane sums a row in column order in the ring as on tiles: the same bits; the oracle to the rounding of
    FP32 factors (nine sweeps of up to 13 terms, 1e-5)."""
    A = getattr(synth, gen)(*size, seed=4)
    n = len(A[0]) - 1
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    slices = -(-n // 32)
    assert n % 32 and slices >= 64 * sms and slices > 2 * unit * 32 * sms and (unit == 1 or slices % unit)
    F = silu.ilu_setup(ctx, silu.Matrix(ctx, *A), kind, 0.0, fill, prec=silu.FP32)
    L, U = F.export()["L"], F.export()["Us"]
    longest = max(int(np.diff(L[0]).max()), int(np.diff(U[0]).max()))
    assert {4: 0, 2: 4, 1: 8}[unit] < longest <= {4: 4, 2: 8, 1: 16}[unit]
    b, x0 = synth.rhs(n, 1, seed=1), synth.rhs(n, 1, seed=2)
    out = []
    for variant in (0, 2):
        F.set_kernel(variant)
        x = dev(x0)
        silu.ilu_smooth(F, x, dev(b), 5, 6)
        ctx.check()
        out.append(host(x))
    assert np.array_equal(out[0], out[1])
    S = oracle.row_scale(oracle.factor(A, kind, 0.0, fill))
    assert relerr(out[0], oracle.smooth(A, S, x0, b, 5, 6)) < 1e-5


@pytest.mark.parametrize("span", [65534, 65535], ids=["widest 16-bit", "narrowest int32"])
def test_columns_at_the_limit_of_16_bits(silu, ctx, span):
    """A slice of 32 rows coupled `up` and `down` rows away spans up + down + 31 columns."""
    n, up = 65800, 32752
    down = span - 31 - up
    i = np.arange(n)
    r = np.concatenate([i, i[:-up], i[down:]])
    c = np.concatenate([i, i[up:], i[:-down]])
    order = np.lexsort((c, r))
    r, c = r[order], c[order]
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, r + 1, 1)
    A = np.cumsum(rp), c.astype(np.int32), np.where(r == c, 4.0, -synth.uniform(5, 1, len(r), 0.1, 1.0))
    lo, hi = np.minimum.reduceat(c, A[0][:-1:32]), np.maximum.reduceat(c, A[0][:-1:32])
    assert (hi - lo).max() == span
    M = silu.Matrix(ctx, *A)
    for nrhs in (1, 2, 3, 4):
        b, x = synth.rhs(n, nrhs, seed=21), synth.rhs(n, nrhs, seed=22)
        out = dev(np.zeros((n, nrhs)))
        M.residual(out, dev(x), dev(b))
        assert maxabs_err(host(out), oracle.residual(A, x, b)) < FP64_TOL, nrhs


# on 152 SMs: 54 to 74 slices per SM, where slices are dealt evenly to the blocks or give way to the tiles
LINES = [("cutcell7", "ilu0", (64, 65, 63)), ("cutcell7", "ilu0", (71, 70, 69)), ("cutcell7", "ilut", (64, 65, 63)),
         ("hex27", "ilu0", (65, 64, 65)), ("hex27", "ilu0", (71, 70, 69))]


@pytest.mark.parametrize("gen,kind,size", LINES, ids=[f"{g}-{k}-{'x'.join(map(str, s))}" for g, k, s in LINES])
def test_both_sides_of_the_lines_match_the_lanes_per_row_kernel(silu, ctx, gen, kind, size):
    """Sums of at most 28 terms of a scaled system, five sweeps: rounding of order 1e-14 (FP32 1e-5)."""
    A = getattr(synth, gen)(*size, seed=6)
    n = len(A[0]) - 1
    M = silu.Matrix(ctx, *A)
    for nrhs in (1, 2, 3, 4):
        b, x0 = synth.rhs(n, nrhs, seed=7), synth.rhs(n, nrhs, seed=8)
        r = dev(np.zeros((n, nrhs)))
        M.residual(r, dev(x0), dev(b))
        assert maxabs_err(host(r), oracle.residual(A, x0, b)) < FP64_TOL, nrhs
    for prec, tol in ((silu.FP64, FP64_TOL), (silu.FP32, 1e-5)):
        F = silu.ilu_setup(ctx, M, kind, 1e-3, 10, prec=prec)
        for nrhs in (1, 2, 3, 4):
            b, x0 = synth.rhs(n, nrhs, seed=7), synth.rhs(n, nrhs, seed=8)
            out = []
            for variant, fused in ((0, 0), (1, 1)):
                F.set_kernel(variant)
                F.set_fused(fused)
                x = dev(x0)
                silu.ilu_smooth(F, x, dev(b), 3, 3)
                ctx.check()
                out.append(host(x))
            assert max(relerr(out[0][:, k], out[1][:, k]) for k in range(nrhs)) < tol, (prec, nrhs)
