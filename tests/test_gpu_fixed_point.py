"""The FP64 kernels that compute in two-limb fixed point (fx.cuh): range and
edge cases of the representation.

Scaling a problem by a power of two only shifts the exponents, so results scale
exactly as long as the exponents stay inside the fixed-point range; outside of
it, and with values that are not finite, the kernels take their FP64 form.
Tolerances as in test_gpu_parity.py (one smoothing step 1e-10)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import workload  # noqa: E402
from oracle import assemble, smoothers  # noqa: E402
from oracle.patches import LocalSolvers  # noqa: E402


@pytest.fixture(scope="module")
def bh():
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device: the -m gpu tests need a GB300")
    import paper_2412_05082_gb300 as m
    m.load()
    return m


def cuda(v):
    return torch.tensor(np.asarray(v), dtype=torch.float64, device="cuda")


def smooth(bh, d, k, L, x, b, tile=0):
    with bh.Context(bh.default_params(d, k, L)) as ctx:
        ctx.set_tile(tile)
        X = x.clone()
        ctx.smooth(L, X, b, 1)
        torch.cuda.synchronize()
        return X


# (degree, level, tile): tile > 0 takes the throughput form at any size, with
# tiles of one patch, a remainder, and more patches than a block takes at once
FORMS = [(2, 3, 0), (2, 4, 32), (3, 4, 7), (4, 4, 0), (4, 4, 17), (5, 4, 3), (6, 4, 0), (7, 4, 8)]


@pytest.mark.parametrize("k,L,tile", FORMS)
def test_smoothing_step_scales_exactly_with_powers_of_two(bh, k, L, tile):
    n = (k * 2 ** L - 1) ** 2
    x, b = cuda(workload.vector_uniform(n, 1)), cuda(workload.rhs_uniform(n, 2))
    ref = smooth(bh, 2, k, L, x, b, tile)
    for s in (-300, -1, 500):
        got = smooth(bh, 2, k, L, x * 2.0 ** s, b * 2.0 ** s, tile)
        assert torch.equal(got, ref * 2.0 ** s), s
    # beyond the fixed-point exponents: the FP64 form, equal up to rounding
    got = smooth(bh, 2, k, L, x * 2.0 ** 720, b * 2.0 ** 720, tile) * 2.0 ** -720
    assert float((got - ref).abs().max()) <= 1e-10 * float((ref - x).abs().max())


@pytest.mark.parametrize("k,L,tile", FORMS)
def test_smoothing_step_with_zero_and_with_wide_inputs(bh, k, L, tile):
    """x = b = 0 stays zero, x = 0 gives the patch solves of b alone, and a
    vector whose patches differ by 2^80 in size is smoothed patch by patch."""
    n1 = k * 2 ** L - 1
    n = n1 * n1
    zero = torch.zeros(n, dtype=torch.float64, device="cuda")
    assert torch.equal(smooth(bh, 2, k, L, zero, zero, tile), zero)
    A = assemble.c0ip_matrix(2, k, 2 ** L)
    loc = LocalSolvers(assemble.c0ip_matrix(2, k, 2 ** L, mixed=False), 2, k, 2 ** L)
    ramp = np.repeat(2.0 ** np.linspace(-40, 40, n1), n1)
    for x, b in ((np.zeros(n), workload.rhs_uniform(n, 3)),
                 (workload.vector_uniform(n, 4) * ramp, workload.rhs_uniform(n, 5) * ramp)):
        ref = smoothers.mvs_step(A, loc, b, x, 1.0)
        got = smooth(bh, 2, k, L, cuda(x), cuda(b), tile).cpu().numpy()
        for row in range(n1):  # every mesh row against its own size
            s = slice(row * n1, (row + 1) * n1)
            lo, hi = max(0, (row - 2 * k) * n1), min(n, (row + 2 * k + 1) * n1)
            assert np.abs(got[s] - ref[s]).max() <= 1e-10 * np.abs(ref - x)[lo:hi].max(), row


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("tile", [0, 5])
def test_values_that_are_not_finite_spread_as_in_fp64(bh, bad, tile):
    """The nodes that a NaN or an infinity in x reaches are those of the
    sequential sweep in FP64."""
    k, L = 3, 4
    n = (k * 2 ** L - 1) ** 2
    A = assemble.c0ip_matrix(2, k, 2 ** L)
    loc = LocalSolvers(assemble.c0ip_matrix(2, k, 2 ** L, mixed=False), 2, k, 2 ** L)
    b = workload.rhs_uniform(n, 6)
    x = workload.vector_uniform(n, 7)
    x[n // 2 + 3] = bad
    got = smooth(bh, 2, k, L, cuda(x), cuda(b), tile).cpu().numpy()
    y = x.copy()
    with np.errstate(invalid="ignore"):
        for v in smoothers.mvs_order(2, 2 ** L):
            I = loc.dofs(v)
            r = b[I] - A[I] @ y
            y[I] = y[I] + loc.solve(v, r) if np.isfinite(r).all() else np.nan
    assert np.array_equal(np.isfinite(got), np.isfinite(y))
    ok = np.isfinite(y)
    assert np.abs(got[ok] - y[ok]).max() <= 1e-10 * np.abs(y[ok] - x[ok]).max()


@pytest.mark.parametrize("d,k,L", [(2, 4, 3), (2, 7, 2), (3, 3, 2), (3, 7, 1)])
def test_exact_solver_scales_exactly_and_spreads_nan(bh, d, k, L):
    """The exact local solver's sliced product: inner lengths from 49 to 2197
    (two parts), tiles of one column, columns scaled by powers of two down to
    denormals, and a NaN that reaches every node of the patches around it."""
    n = (k * 2 ** L - 1) ** d

    def step(x, b):
        with bh.Context(bh.default_params(d, k, L, local_solver=bh.EXACT)) as ctx:
            X = x.clone()
            ctx.smooth(L, X, b, 1)
            torch.cuda.synchronize()
            return X

    x, b = cuda(workload.vector_uniform(n, 8)), cuda(workload.rhs_uniform(n, 9))
    ref = step(x, b)
    for s in (-400, 3, 500):
        assert torch.equal(step(x * 2.0 ** s, b * 2.0 ** s), ref * 2.0 ** s), s
    zero = torch.zeros_like(b)
    tiny = step(zero, b * 2.0 ** -1015) * 2.0 ** 1015
    assert float((tiny - step(zero, b)).abs().max()) <= 1e-2 * float(tiny.abs().max())
    b[0] = float("nan")
    assert bool(torch.isnan(step(x, b)[0]))


@pytest.mark.parametrize("d,k,L", [(2, 2, 7), (2, 3, 2), (2, 4, 1), (2, 7, 3), (3, 3, 1), (3, 4, 2), (3, 7, 2)])
def test_operator_scales_exactly_and_spreads_nan(bh, d, k, L):
    """apply_A and the residual in fixed point: exact under powers of two,
    zero lines, the FP64 form beyond the exponents, and a NaN that reaches the
    rows that couple to it and no others than its band."""
    n1 = k * 2 ** L - 1
    n = n1 ** d
    x, b = cuda(workload.vector_uniform(n, 11)), cuda(workload.rhs_uniform(n, 12))
    with bh.Context(bh.default_params(d, k, L)) as ctx:
        def residual(x, b):
            r = torch.empty_like(x)
            ctx.residual(L, x, b, r)
            torch.cuda.synchronize()
            return r
        ref = residual(x, b)
        for s in (-300, 1, 400):
            assert torch.equal(residual(x * 2.0 ** s, b * 2.0 ** s), ref * 2.0 ** s), s
        big = residual(x * 2.0 ** 720, b * 2.0 ** 720) * 2.0 ** -720
        assert float((big - ref).abs().max()) <= 1e-12 * float(ref.abs().max())
        zero = torch.zeros_like(x)
        assert torch.equal(residual(zero, b), b)
        if n > 3000:
            return
        A = assemble.c0ip_matrix(d, k, 2 ** L)
        x[n // 2] = float("nan")
        got = torch.isnan(residual(x, b)).cpu().numpy()
        assert np.all(got[(A[:, n // 2].toarray().ravel() != 0)])
        assert got.sum() <= (4 * k + 1) ** d


@pytest.mark.parametrize("k,tile", [(2, 32), (3, 9), (4, 17), (5, 5), (6, 9), (7, 8)])
def test_requested_tile_takes_the_throughput_form(bh, k, tile):
    """A tile that is asked for is computed by the throughput form on any level, so
    that small problems reach it: its scales and folded lines round differently from
    the latency form that a level with few patches takes by itself, to the same
    result; and it hands patches over to the FP64 form."""
    L = 4
    n1 = k * 2 ** L - 1
    n = n1 * n1
    A = assemble.c0ip_matrix(2, k, 2 ** L)
    loc = LocalSolvers(assemble.c0ip_matrix(2, k, 2 ** L, mixed=False), 2, k, 2 ** L)
    x, b = workload.vector_uniform(n, 21), workload.rhs_uniform(n, 22)
    ref = smoothers.mvs_step(A, loc, b, x, 1.0)
    small = smooth(bh, 2, k, L, cuda(x), cuda(b), 0)
    got = smooth(bh, 2, k, L, cuda(x), cuda(b), tile)
    assert not torch.equal(got, small)
    for v in (got, small):
        assert np.abs(v.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref - x).max()
    # one value out of range: the patches around it in FP64, the others of their tiles
    # unchanged (the middle of the domain, all patches there away from the boundary)
    far = x.copy()
    far[n // 2] = 2.0 ** 800
    hit = smooth(bh, 2, k, L, cuda(far), cuda(b), tile).cpu().numpy()
    assert np.isfinite(hit).all()
    assert np.array_equal(hit[:k], got.cpu().numpy()[:k])
    far[n // 2] = np.nan
    hit = smooth(bh, 2, k, L, cuda(far), cuda(b), tile).cpu().numpy()
    assert np.isnan(hit[n // 2]) and np.isfinite(hit[:k]).all()


@pytest.mark.parametrize("k,gamma", [(2, 1.0), (2, 1.04), (2, 1.2), (2, 60.0), (3, 5.0), (4, 500.0)])
@pytest.mark.parametrize("tile", [0, 6])
def test_penalties_that_leave_negative_eigenvalues(bh, k, gamma, tile):
    """A penalty below the default can leave the 1D patch matrices at the boundary
    indefinite (negative eigenvalues at Q2 with 1.0 to 1.2) while the coarse matrix
    is positive definite; larger ones widen the spectrum."""
    L = 3
    n = (k * 2 ** L - 1) ** 2
    A = assemble.c0ip_matrix(2, k, 2 ** L, gamma)
    loc = LocalSolvers(assemble.c0ip_matrix(2, k, 2 ** L, gamma, mixed=False), 2, k, 2 ** L)
    x, b = workload.vector_uniform(n, 31), workload.rhs_uniform(n, 32)
    ref = smoothers.mvs_step(A, loc, b, x, 1.0)
    with bh.Context(bh.default_params(2, k, L, gamma=gamma)) as ctx:
        ctx.set_tile(tile)
        X = cuda(x)
        ctx.smooth(L, X, cuda(b), 1)
        got = X.cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref - x).max()
