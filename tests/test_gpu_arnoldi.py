"""The Arnoldi step of FGMRES at the edges of its forms: one cluster of 1, 2
and 16 blocks, a launch per basis vector (between the forms and above them),
and grids of one, two and three groups of rows per block, against flexible
GMRES in plain torch on the library's products and smoother."""
import math

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def silu():
    import paper_2111_09512_gb300 as s
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s.build()
    return s


def fgmres(silu, M, F, b, restart, its, sweeps):
    """`its` iterations in cycles of `restart` from zero (modified Gram-Schmidt, one least-squares solve per cycle)."""
    zero = torch.zeros_like(b)

    def mul(v):
        r = torch.empty_like(v)
        M.residual(r, v, zero)
        return -r

    x = torch.zeros_like(b)
    while its > 0:
        r = b - mul(x)
        beta = r.norm()
        V, Z = [r / beta], []
        m = min(restart, its)
        H = torch.zeros(m + 1, m, dtype=torch.float64)
        for j in range(m):
            z = torch.zeros_like(b)
            silu.ilu_smooth(F, z, V[j], *sweeps)
            w = mul(z)
            for i in range(j + 1):
                h = torch.dot(w, V[i])
                w = w - h * V[i]
                H[i, j] = h.cpu()
            H[j + 1, j] = w.norm().cpu()
            V.append(w / w.norm())
            Z.append(z)
        rhs = torch.zeros(m + 1, 1, dtype=torch.float64)
        rhs[0] = beta.cpu()
        y = torch.linalg.lstsq(H, rhs).solution[:, 0]
        for j in range(m):
            x = x + y[j].item() * Z[j]
        its -= m
    return x, ((b - mul(x)).norm() / b.norm()).item()


# rows / 2048, rounded up: 1, 2, 16, 17, 151, 152, 250, 307, 455, 460
SIZES = [(13, 11, 9), (16, 16, 8), (17, 11, 11), (32, 32, 32), (33, 31, 33), (68, 67, 67), (68, 68, 67), (80, 80, 80),
         (86, 86, 85), (98, 98, 97), (98, 98, 98)]


@pytest.mark.parametrize("size", SIZES, ids=["x".join(map(str, s)) for s in SIZES])
def test_arnoldi_step_matches_plain_fgmres(silu, size):
    ctx = silu.Context(0, torch.cuda.current_stream())
    A = synth.poisson7(*size)
    n = len(A[0]) - 1
    M = silu.Matrix(ctx, *A)
    F = silu.ilu_setup(ctx, M, "ilu0")
    b = torch.from_numpy(synth.rhs(n, 1, seed=3)[:, 0]).cuda()
    for restart, its in ((7, 10), (30, 12)):
        want, rel = fgmres(silu, M, F, b, restart, its, (3, 3))
        x = torch.zeros_like(b)
        for _ in range(2):  # captured on the first solve, replayed on the second
            x.zero_()
            st, done, relres = silu.fgmres_solve(F, x, b, tol=0.0, restart=restart, maxit=its, sweeps_L=3, sweeps_U=3)
            ctx.check()
            assert st == silu.ERR_NOT_CONVERGED and done == its
            # Krylov iterates of a well-conditioned start: rounding (1e-16) times a modest growth
            assert ((x - want).norm() / want.norm()).item() < 1e-10
            assert math.isclose(relres, rel, rel_tol=1e-6)


def test_arnoldi_grids_of_several_streams_run_side_by_side(silu):
    """Solves on four streams from four host threads, each a grid of resident
    blocks per iteration, give the bits they give alone."""
    import threading
    sizes = [(80, 80, 80), (98, 98, 97), (86, 86, 85), (32, 32, 32)]
    jobs = []
    for k, size in enumerate(sizes):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            ctx = silu.Context(0, stream)
            A = synth.poisson7(*size)
            n = len(A[0]) - 1
            F = silu.ilu_setup(ctx, silu.Matrix(ctx, *A), "ilu0")
            b = torch.from_numpy(synth.rhs(n, 1, seed=k)[:, 0]).cuda()
            jobs.append((ctx, F, b, torch.zeros_like(b), stream))
    torch.cuda.synchronize()

    def solve(job, reps):
        ctx, F, b, x, stream = job
        torch.cuda.set_device(0)
        with torch.cuda.stream(stream):
            for _ in range(reps):
                x.zero_()
                st, its, rel = silu.fgmres_solve(F, x, b, tol=0.0, restart=30, maxit=40, sweeps_L=3, sweeps_U=3)
                assert st == silu.ERR_NOT_CONVERGED and its == 40
            ctx.check()

    alone = []
    for job in jobs:
        solve(job, 1)
        torch.cuda.synchronize()
        alone.append(job[3].clone())
    failed = []

    def run(job):
        try:
            solve(job, 6)
        except BaseException as e:  # reported by the main thread
            failed.append(e)

    threads = [threading.Thread(target=run, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    torch.cuda.synchronize()
    for job, want in zip(jobs, alone):
        assert torch.equal(job[3], want)


@pytest.mark.parametrize("size", [(32, 32, 32), (68, 68, 67), (98, 98, 97)], ids=["cluster", "one group", "three groups"])
def test_solve_after_a_step_that_gave_up(silu, size):
    """A wait of the exchange that runs out is reported; entries it leaves, numbered like the next solve's, are not
    read by that solve, which gives the bits of one before."""
    ctx = silu.Context(0, torch.cuda.current_stream())
    A = synth.poisson7(*size)
    n = len(A[0]) - 1
    F = silu.ilu_setup(ctx, silu.Matrix(ctx, *A), "ilu0")
    b = torch.from_numpy(synth.rhs(n, 1, seed=3)[:, 0]).cuda()
    out = []
    for gave_up in (False, True, True):
        if gave_up:
            F.selftest_exchange()
            with pytest.raises(silu.SiluError) as e:
                ctx.check()
            assert e.value.status == silu.ERR_TIMEOUT
        x = torch.zeros_like(b)
        st, its, _ = silu.fgmres_solve(F, x, b, tol=0.0, restart=5, maxit=12, sweeps_L=3, sweeps_U=3)
        ctx.check()
        assert st == silu.ERR_NOT_CONVERGED and its == 12
        out.append(x)
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])


def division_operands():
    """(w, h): mantissas at random, all ones, next to powers of two and of few bits, with exponents on both sides of
    the limits of the short division (2^+-300 of the divisor, 2^+-600 of the dividend), and the special values."""
    rng = np.random.RandomState(5)

    def mantissas(count):
        m = rng.randint(0, 2**52, count, dtype=np.int64)
        kind = rng.randint(0, 6, count)
        m[kind == 1] = 2**52 - 1 - rng.randint(0, 4, (kind == 1).sum())
        m[kind == 2] = rng.randint(0, 4, (kind == 2).sum())
        m[kind == 3] &= -(1 << 40)
        return m

    def doubles(m, e):
        return ((np.asarray(e, np.int64) + 1023 << 52) | m | (rng.randint(0, 2, len(m)).astype(np.int64) << 63)).view(
            np.float64)

    n = 1 << 21
    out = [(doubles(mantissas(n), rng.randint(-40, 41, n)), doubles(mantissas(n), rng.randint(-40, 41, n)))]
    edge_w, edge_h = np.array([-601, -600, -599, 598, 599, 600, 601]), np.array([-301, -300, -299, 298, 299, 300, 301])
    out.append((doubles(mantissas(n), rng.choice(edge_w, n)), doubles(mantissas(n), rng.choice(edge_h, n))))
    out.append((doubles(mantissas(n), rng.randint(-1022, 1024, n)), doubles(mantissas(n), rng.randint(-1022, 1024, n))))
    special = np.array([0.0, -0.0, 5e-324, -5e-324, 2.2250738585072009e-308, 2.2250738585072014e-308, 1.0, -3.0, 1e308,
                        1.7976931348623157e308, np.inf, -np.inf, np.nan])
    special = np.concatenate([special, doubles(mantissas(40), rng.randint(-1022, 1024, 40))])
    w, h = np.meshgrid(special, special)
    out.append((w.ravel(), h.ravel()))
    return out


def test_division_of_the_normalisation_is_correctly_rounded(silu):
    ctx = silu.Context(0, torch.cuda.current_stream())
    for w, h in division_operands():
        wd, hd = torch.from_numpy(w.copy()).cuda(), torch.from_numpy(h.copy()).cuda()
        q = torch.empty_like(wd)
        ctx.selftest_divide(wd, hd, q)
        ctx.check()
        with np.errstate(all="ignore"):
            want = w / h
        got = q.cpu().numpy()
        nan = np.isnan(want)
        assert np.isnan(got[nan]).all()
        assert np.array_equal(got[~nan].view(np.int64), want[~nan].view(np.int64))
