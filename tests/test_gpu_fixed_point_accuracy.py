"""How accurate the FP64 kernels that compute in two-limb fixed point (fx.cuh) are
where values of one line or patch differ in size, and at a smooth solution.

References are in numpy's long double, with the 1D matrices that the library
builds.  Tolerances are what FP64 arithmetic itself guarantees or does: for the
operator, row by row, the a-priori bound of a chain of FP64 sums; for a patch
step, that bound carried through the inverse of the patch, and the movement that
the same sums in FP64 cause."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LD = np.longdouble
U = 2.0 ** -53


@pytest.fixture(scope="module")
def bh():
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device: the -m gpu tests need a GB300")
    import paper_2412_05082_gb300 as m
    m.load()
    return m


def cuda(v):
    return torch.tensor(np.asarray(v, dtype=np.float64).ravel(), device="cuda")


def line_matrices(bh, k, N):
    """M, L, B of a line of N >= 4 unit cells from the rows of a line of 7, which
    are the library's tables."""
    out = []
    for which in range(3):
        P = bh.setup_1d(k, k * (k + 1.0), 7, which)
        A = np.zeros((k * N + 1, k * N + 1))
        for g in range(1, k * N):
            src = g if g <= k else (7 * k - (k * N - g) if g >= k * N - k else 3 * k + g % k)
            for t in range(-2 * k, 2 * k + 1):
                if 0 <= src + t <= 7 * k and 0 <= g + t <= k * N:
                    A[g, g + t] = P[src, src + t]
        out.append(A[1:-1, 1:-1])
    return out


def terms(d, mats):
    """(factor, matrix per axis, x first) of the Kronecker form."""
    M, L, B = mats
    if d == 2:
        return [(1, (M, B)), (2, (L, L)), (1, (B, M))]
    return [(1, (B, M, M)), (1, (M, B, M)), (1, (M, M, B)),
            (2, (L, L, M)), (2, (L, M, L)), (2, (M, L, L))]


def along(P, x, axis):
    """P applied along an axis of x, by its bands."""
    x = np.moveaxis(x, axis, -1)
    y = np.zeros(x.shape[:-1] + (P.shape[0],), dtype=x.dtype)
    P = P.astype(x.dtype)
    for g in range(P.shape[0]):
        nz = np.flatnonzero(P[g])
        for j in nz:  # one term after the other, as the kernels sum
            y[..., g] = y[..., g] + P[g, j] * x[..., j]
    return np.moveaxis(y, -1, axis)


def apply(d, mats, x):
    """The operator on an array of d axes, the last one x."""
    y = 0
    for f, ops in terms(d, mats):
        t = x
        for a in range(d):
            t = along(ops[a], t, d - 1 - a)
        y = y + f * t
    return y


def graded(kind, shape, at, rng):
    """Uniform values times a field that changes by many powers of two."""
    x = rng.uniform(-1, 1, shape)
    n = shape[-1]
    if kind == "spike":
        x[tuple(min(at, m - 1) for m in shape)] = 2.0 ** 70
    elif kind == "jump":
        x[..., at:] *= 2.0 ** 30
    elif kind == "jump_last":
        x[at:] *= 2.0 ** 30
    else:
        x *= 2.0 ** np.linspace(-80, 80, n)
    return x


# the spike and the jumps at every cell of a block of four cells
@pytest.mark.parametrize("d,k,L", [(2, 3, 4), (2, 4, 3), (2, 7, 3), (3, 3, 3), (3, 5, 2)])
@pytest.mark.parametrize("kind", ["spike", "jump", "jump_last", "ramp"])
def test_operator_rows_are_accurate_to_their_own_values(bh, d, k, L, kind):
    """Every row of A x and of b - A x within n u sum |a_ij| |x_j|, n the roundings
    of a chain of FP64 sums, wherever larger values lie on the line."""
    N = 2 ** L
    n = k * N - 1
    mats = line_matrices(bh, k, N)
    absm = [np.abs(m) for m in mats]
    rng = np.random.default_rng(10 * k + d)
    tol = (d * (4 * k + 2) + 6) * U
    with bh.Context(bh.default_params(d, k, L)) as ctx:
        for cell in range(0, 4 if kind != "ramp" else 1):
            x = graded(kind, (n,) * d, k * cell + cell % k, rng)
            X, Y = cuda(x), torch.empty(n ** d, dtype=torch.float64, device="cuda")
            ctx.apply_A(L, X, Y)
            scale = float(N) ** (4 - d)
            y = Y.cpu().numpy().reshape(x.shape)
            ref = apply(d, mats, x.astype(LD)) * LD(scale)
            size = (apply(d, absm, np.abs(x)) * scale)
            assert (np.abs((y - ref).astype(np.float64)) <= tol * size).all(), cell
            b = np.ldexp(rng.uniform(-1, 1, x.shape), np.frexp(size)[1])
            ctx.residual(L, X, cuda(b), Y)
            r = Y.cpu().numpy().reshape(x.shape)
            err = np.abs((r - (b.astype(LD) - ref)).astype(np.float64))
            assert (err <= tol * (size + np.abs(b))).all(), cell


def color0_patches(k, N):
    """(x slice, y slice, vertex) of the patches of color 0."""
    m = 2 * k - 1
    for vy in range(2, N, 2):
        for vx in range(2, N, 2):
            if (vx // 2 + vy // 2) % 2 == 0:
                yield slice(k * (vx - 1), k * (vx - 1) + m), slice(k * (vy - 1), k * (vy - 1) + m)


def local_matrix(mats, sx, sy):
    M, L, B = mats
    return np.kron(B[sy, sy], M[sx, sx]) + np.kron(M[sy, sy], B[sx, sx])


@pytest.mark.parametrize("tile", [0, 5])
@pytest.mark.parametrize("k", [3, 4, 6, 7])
def test_step_at_a_smooth_solution_moves_it_no_further_than_fp64(bh, k, tile):
    """One color at a smooth solution (b = A x in long double): what moves it is the
    rounding of the residual, which in FP64 sums is the measure."""
    L, N = 4, 16
    n = k * N - 1
    mats = line_matrices(bh, k, N)
    s = np.sin(np.pi * np.linspace(0, 1, n + 2)[1:-1]) ** 2
    x = np.outer(s, s) * (1 + 0.3 * np.outer(s, s[::-1]))
    b = apply(2, mats, x.astype(LD)).astype(np.float64)
    with bh.Context(bh.default_params(2, k, L)) as ctx:
        ctx.set_tile(tile)
        X = cuda(x)
        ctx.smooth_colors(L, X, cuda(b * float(N) ** 2), 0, 1)
        got = X.cpu().numpy().reshape(n, n) - x
    r64 = b - apply(2, mats, x)
    moved = fp64 = 0.0
    for sx, sy in color0_patches(k, N):
        A = local_matrix(mats, sx, sy)
        moved += (got[sy, sx] ** 2).sum()
        fp64 += (np.linalg.solve(A, r64[sy, sx].ravel()) ** 2).sum()
    assert moved <= fp64, (np.sqrt(moved), np.sqrt(fp64))


@pytest.mark.parametrize("tile", [0, 5])
@pytest.mark.parametrize("k", [2, 4, 7])
@pytest.mark.parametrize("kind", ["spike", "jump", "jump_last", "ramp"])
def test_step_at_a_graded_solution_is_accurate_patch_by_patch(bh, k, kind, tile):
    """One color at solutions that change by 2^30 and more over a few nodes: every
    patch moves by less than FP64's bound for its own residual (n u sum |a_ij| |x_j|)
    carried through the inverse of the patch."""
    L, N = 4, 16
    n = k * N - 1
    mats = line_matrices(bh, k, N)
    absm = [np.abs(m) for m in mats]
    rng = np.random.default_rng(k)
    tol = (2 * (4 * k + 2) + 6 + 4 * (2 * k - 1)) * U
    with bh.Context(bh.default_params(2, k, L)) as ctx:
        ctx.set_tile(tile)
        for at in (k * 8 - 1, k * 8 + k // 2, k * 9 - 1):
            x = graded(kind, (n, n), at, rng)
            b = apply(2, mats, x.astype(LD)).astype(np.float64)
            size = apply(2, absm, np.abs(x))
            X = cuda(x)
            ctx.smooth_colors(L, X, cuda(b * float(N) ** 2), 0, 1)
            got = np.abs(X.cpu().numpy().reshape(n, n) - x)
            for sx, sy in color0_patches(k, N):
                inv = np.abs(np.linalg.inv(local_matrix(mats, sx, sy)))
                bound = tol * (inv @ size[sy, sx].ravel()) + U * np.abs(x[sy, sx]).ravel()
                assert (got[sy, sx].ravel() <= bound).all(), (at, sx.start, sy.start)


@pytest.mark.parametrize("d,k", [(2, 4), (2, 7), (3, 3), (3, 4)])
def test_exact_solver_keeps_every_entry_of_its_inverse(bh, d, k):
    """On the single patch of level 1 the correction of a unit vector is a column of
    the patch inverse, a symmetric matrix: entry (i, j) from column j and entry (j, i)
    from column i agree to rounding, however much smaller than the largest entry of
    its row it is."""
    n = (2 * k - 1) ** d
    Y = np.empty((n, n))
    with bh.Context(bh.default_params(d, k, 1, local_solver=bh.EXACT)) as ctx:
        x = torch.empty(n, dtype=torch.float64, device="cuda")
        b = torch.zeros(n, dtype=torch.float64, device="cuda")
        for j in range(n):
            x.zero_()
            b.zero_()
            b[j] = 1.0
            ctx.smooth(1, x, b, 1)
            Y[j] = x.cpu().numpy()
    assert (np.abs(Y - Y.T) <= 4 * U * np.abs(Y)).all()
