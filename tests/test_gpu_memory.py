"""Device memory that runs out: the failing call says so, and the objects stay
usable (allocations fail on the host side, silu_selftest_memory)."""
import numpy as np
import pytest

import oracle
import synth
from _helpers import relerr

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


@pytest.fixture
def limit(silu):
    """Call with a number of bytes in use that may not be exceeded; lifted at the end."""
    yield silu.silu_selftest_memory
    silu.silu_selftest_memory(-1)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def out_of_memory(silu, call):
    with pytest.raises(silu.SiluError) as e:
        call()
    assert e.value.status == silu.ERR_OOM


SHAPE = (21, 19, 17)


def test_smaller_requests_after_a_workspace_that_did_not_fit(silu, limit):
    """Growing a workspace releases its buffers one by one: after a failure in the middle a request that the old
    workspace would have held is allocated anew."""
    ctx = silu.Context(0, torch.cuda.current_stream())
    A = synth.cutcell7(*SHAPE, seed=2)
    n = len(A[0]) - 1
    F = silu.ilu_setup(ctx, silu.Matrix(ctx, *A), "ilu0")
    S = oracle.row_scale(oracle.factor(A, "ilu0", 0.0, 0))
    b4, b64 = synth.rhs(n, 4, seed=1), synth.rhs(n, 64, seed=2)

    def smooth(b):
        x = dev(np.zeros_like(b))
        silu.ilu_smooth(F, x, dev(b), 3, 3)
        return host(x)

    smooth(b4)
    want = oracle.smooth(A, S, np.zeros_like(b4), b4, 3, 3)
    used = silu.silu_selftest_memory()  # a buffer that has grown keeps its size: limits are counted from here
    # 64 columns take 512 bytes a row in each of four vectors, where 32 are released each time
    for more in (0, 500 * n, 1000 * n, 1500 * n):
        limit(used + more)
        out_of_memory(silu, lambda: smooth(b64))
        silu.silu_selftest_memory(-1)
        assert relerr(smooth(b4), want) < FP64_TOL, more
    b = dev(b4[:, 0])

    def solve(restart):
        x = torch.zeros_like(b)
        st, its, _ = silu.fgmres_solve(F, x, b, tol=0.0, restart=restart, maxit=9, sweeps_L=2, sweeps_U=2)
        ctx.check()
        assert st == silu.ERR_NOT_CONVERGED and its == 9
        return host(x)

    before = solve(7)
    used = silu.silu_selftest_memory()
    for more in (0, 950 * n, 1400 * n):  # 121 and 120 vectors of 8 bytes a row, where 8 and 7 are released
        limit(used + more)
        out_of_memory(silu, lambda: solve(120))
        silu.silu_selftest_memory(-1)
        assert np.array_equal(solve(7), before), more


def test_smaller_restart_after_a_batch_workspace_that_did_not_fit(silu, limit):
    ctx = silu.Context(0, torch.cuda.current_stream())
    B = silu.Batch(ctx, [synth.cutcell7(e, e, e, seed=e) for e in (9, 12, 15)], "ilu0")
    b = dev(synth.rhs(B.n, 1, seed=3)[:, 0])

    def solve(restart):
        x = torch.zeros_like(b)
        silu.silu_batch_fgmres(B, x, b, tol=0.0, restart=restart, maxit=9, sweeps_L=2, sweeps_U=2)
        ctx.check()
        return host(x)

    before = solve(7)
    used = silu.silu_selftest_memory()
    for more in (0, 950 * B.n, 1400 * B.n):
        limit(used + more)
        out_of_memory(silu, lambda: solve(120))
        silu.silu_selftest_memory(-1)
        assert np.array_equal(solve(7), before), more


def test_tiles_stay_in_place_when_new_ones_do_not_fit(silu, limit):
    ctx = silu.Context(0, torch.cuda.current_stream())
    A = synth.cutcell7(*SHAPE, seed=2)
    n = len(A[0]) - 1
    M = silu.Matrix(ctx, *A)
    M.set_shape(1, 1, 16)
    b, x = dev(synth.rhs(n, 1, seed=4)), dev(synth.rhs(n, 1, seed=5))
    r = torch.zeros_like(b)
    limit(0)
    out_of_memory(silu, lambda: M.set_shape(4, 1, 16))
    M.residual(r, x, b)
    assert relerr(host(r), oracle.residual(A, host(x), host(b))) < FP64_TOL


def every_setup(silu, ctx):
    """One of each object and call that takes device memory, in one context; all results for one right-hand side."""
    A = synth.cutcell7(*SHAPE, seed=2)
    n = len(A[0]) - 1
    b = dev(synth.rhs(n, 1, seed=6)[:, 0])
    out, kept = [], []

    def result(call):
        x = torch.zeros_like(b)
        call(x)
        ctx.check()
        out.append(host(x))

    M = silu.Matrix(ctx, *A)
    F = silu.ilu_setup(ctx, M, "ilu0")
    out.append(F.power_norms("U", 2, 3, synth.rhs(n, 1, seed=7)[:, 0]))
    F.set_direct(1)  # the automatic choice is timed
    result(lambda x: silu.direct_trisolve(F, x, b))
    result(lambda x: silu.ilu_smooth(F, x, b, 3, 3))
    result(lambda x: silu.fgmres_solve(F, x, b, tol=0.0, restart=25, maxit=9, sweeps_L=2, sweeps_U=2))
    F.amg_setup(coarse_size=100, ilu_levels=2)
    result(lambda x: F.amg_vcycle(x, b, 2, 2))
    F.schur_setup(3, 1e-3, 5)
    result(lambda x: F.schur_smooth(x, b, 2, 2))
    G = silu.ilu_setup(ctx, M, "ilut", 1e-3, 10, prec=silu.FP32)
    G.set_direct(2)
    result(lambda x: silu.ilu_smooth(G, x, b, 3, 3))
    result(lambda x: silu.direct_trisolve(G, x, b))
    result(lambda x: silu.fgmres_solve(F, x, b, tol=0.0, restart=25, maxit=9, sweeps_L=2, sweeps_U=2))
    B = silu.Batch(ctx, [A, synth.cutcell7(9, 9, 9, seed=1)], "ilu0")
    bb = dev(synth.rhs(B.n, 1, seed=8)[:, 0])
    xb = torch.zeros_like(bb)
    silu.silu_batch_fgmres(B, xb, bb, tol=0.0, restart=11, maxit=9, sweeps_L=2, sweeps_U=2)
    ctx.check()
    out.append(host(xb))
    silu.ilu_refactor(F, A[2] * 2.0)
    result(lambda x: silu.ilu_smooth(F, x, b, 3, 3))
    kept += [M, F, G, B]
    return out, kept


def test_what_fits_without_sliced_copies_still_fits(silu, limit):
    """Memory for the objects alone: the copies give way in every setup, and results keep their bits."""
    base = silu.silu_selftest_memory()
    ctx = silu.Context(0, torch.cuda.current_stream())
    free, kept = every_setup(silu, ctx)
    with_copies = silu.silu_selftest_memory() - base
    del kept
    ctx = silu.Context(0, torch.cuda.current_stream())
    ctx.set_copies(False)
    bare, kept = every_setup(silu, ctx)
    without = silu.silu_selftest_memory() - base
    assert without < with_copies
    del kept
    ctx = silu.Context(0, torch.cuda.current_stream())
    limit(base + without)
    short, kept = every_setup(silu, ctx)
    for other in (bare, short):
        assert len(other) == len(free)
        assert all(np.array_equal(f, o) for f, o in zip(free, other))


def test_a_workspace_takes_the_memory_of_the_copies(silu, limit):
    """Growth of the workspace by as much as the copies hold, also after an exact solve, whose factors are those of
    the sweeps."""
    ctx = silu.Context(0, torch.cuda.current_stream())
    A = synth.cutcell7(*SHAPE, seed=2)
    n = len(A[0]) - 1
    F = silu.ilu_setup(ctx, silu.Matrix(ctx, *A), "ilu0")
    b = dev(synth.rhs(n, 1, seed=6)[:, 0])
    x = torch.zeros_like(b)
    silu.direct_trisolve(F, x, b)
    F.reserve(1, 20)
    torch.cuda.synchronize()
    limit(silu.silu_selftest_memory())
    # A and two factors, 13 entries a row: copies of at least 10 bytes an entry
    F.reserve(3, 20)  # 4 vectors of 16 bytes a row more
    F.reserve(3, 23)  # 48 bytes a row more


def test_giving_up_the_copies_keeps_results_and_captured_solves(silu):
    ctx = silu.Context(0, torch.cuda.current_stream())
    A = synth.cutcell7(*SHAPE, seed=2)
    n = len(A[0]) - 1
    M = silu.Matrix(ctx, *A)
    F = silu.ilu_setup(ctx, M, "ilu0")
    B = silu.Batch(ctx, [A], "ilu0")
    b = dev(synth.rhs(n, 1, seed=6)[:, 0])
    out = []
    for copies in (True, False):
        ctx.set_copies(copies)
        x, y, r = torch.zeros_like(b), torch.zeros_like(b), torch.zeros_like(b)
        silu.fgmres_solve(F, x, b, tol=0.0, restart=7, maxit=9, sweeps_L=2, sweeps_U=2)
        silu.silu_batch_fgmres(B, y, b, tol=0.0, restart=7, maxit=9, sweeps_L=2, sweeps_U=2)
        M.residual(r, x, b)
        ctx.check()
        out.append((host(x), host(y), host(r)))
    assert all(np.array_equal(p, q) for p, q in zip(*out))
    used = silu.silu_selftest_memory()
    M2 = silu.Matrix(ctx, *A)
    bare = silu.silu_selftest_memory() - used
    ctx.set_copies(True)
    M3 = silu.Matrix(ctx, *A)
    assert silu.silu_selftest_memory() - used > 2 * bare + 10 * 6 * n


@pytest.mark.parametrize("shape", [SHAPE, (258, 257, 2)], ids=["16-bit columns", "int32 columns"])
def test_refactorisation_fills_the_copies_in_place(silu, limit, shape):
    """New values on the same pattern take no memory, and the factors keep their sliced copies."""
    ctx = silu.Context(0, torch.cuda.current_stream())
    A, A2 = synth.cutcell7(*shape, seed=3), synth.cutcell7(*shape, seed=8)
    n = len(A[0]) - 1
    b, x0 = synth.rhs(n, 1, seed=5), synth.rhs(n, 1, seed=6)
    for prec, tol in ((silu.FP64, FP64_TOL), (silu.FP32, 1e-5)):
        F = silu.ilu_setup(ctx, silu.Matrix(ctx, *A), "ilu0", prec=prec)
        F.reserve(1)
        torch.cuda.synchronize()
        used = silu.silu_selftest_memory()
        limit(used)
        silu.ilu_refactor(F, A2[2])
        limit(-1)
        assert silu.silu_selftest_memory() == used
        x = dev(x0)
        silu.ilu_smooth(F, x, dev(b), 4, 4)  # at once: the copies are complete when a sweep starts
        S = oracle.row_scale(oracle.factor(A2, "ilu0", 0.0, 0))
        assert relerr(host(x), oracle.smooth(A2, S, x0, b, 4, 4)) < tol
