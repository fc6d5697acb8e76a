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
