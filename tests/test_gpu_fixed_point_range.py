"""Values at the ends of FP64's range and of uneven magnitude in the block fixed-point element kernels."""
import numpy as np
import pytest
import torch

import paper_2004_06722_gb300 as pkg
from oracle.element import element_matrices
from oracle.basis import lagrange_derivatives, lagrange_values
from oracle.quadrature import bp_rule, gll
from synth import uniform_pm1
from tensor_reference import Element

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    pkg.load_library()


def _run(op, uL):
    return op.bk_apply(torch.from_numpy(np.ascontiguousarray(uL)).cuda()).cpu().numpy()


@pytest.mark.parametrize("bp,N", [(5, 2), (5, 3), (5, 7), (6, 4), (1, 3), (3, 3), (4, 2)])
@pytest.mark.parametrize("k", [-1030, -1045])
def test_subnormal_elements(bp, N, k):
    """An element of subnormal values alone is not an element of zeros (below 2^-1042 a value's upper word
    is zero).  Every rounding of the FP64 form is then within 2^-1075, about a hundred of them times row sums
    below 2^7: 2^-1061 against results of about 2^(k-9), which is 1e-2 of the largest at k = -1045 and
    below 1e-6 at k = -1030."""
    op = pkg.Operator.box(bp, 2, 1, 1, N)
    shape = (2, (N + 1) ** 3) if op.ncomp == 1 else (2, (N + 1) ** 3, 3)
    uL = np.ldexp(np.round(np.ldexp(uniform_pm1(9, np.arange(int(np.prod(shape)))).reshape(shape), 20)), -20)
    uL[1, :] = 0.0
    rule = bp_rule(bp, N)
    which = "B" if bp in (1, 2) else "A"
    ref = element_matrices(op.coords[0], N, rule, want=(which,))[which] @ uL[0]
    w = _run(op, np.ldexp(uL, k))
    assert not w[1].any()
    got = np.ldexp(w[0], -k)
    assert np.abs(got - ref).max() < (1e-2 if k == -1045 else 1e-6) * np.abs(ref).max()


@pytest.mark.parametrize("bp,N", [(5, 1), (5, 2), (6, 1), (6, 2)])
@pytest.mark.parametrize("aspect", [30.0, 1e2, 1e4])
def test_thin_elements(bp, N, aspect):
    """A function of x alone on boxes thin in z: at these orders D takes constants to exact zeros in FP64, so nothing of the small fluxes is lost (A u is a product of 1D sums, about 20 roundings)."""
    coords, l2g, _ = pkg.mesh_box(2, 1, 1, N, 0.0)
    coords = coords * np.array([1.0, 1.0, 1.0 / aspect])
    op = pkg.Operator(bp, N, coords, l2g, None)
    p1 = N + 1
    f = np.array([0.7, -0.4, 0.9])[:p1]
    u = np.tile(f, p1 * p1)
    uL = np.repeat(u[None], 2, 0)
    w = _run(op, uL if op.ncomp == 1 else np.repeat(uL[..., None], 3, -1)).reshape(2, p1 ** 3, -1)
    pts, wq = bp_rule(bp, N)
    J, D = lagrange_values(gll(N)[0], pts), lagrange_derivatives(gll(N)[0], pts)
    a = 4.0 * D.T @ (wq * (D @ f))  # hx = 1/2
    my, mz = 0.5 * J.T @ wq, 0.5 / aspect * J.T @ wq
    ref = np.einsum("k,j,i->kji", mz, my, a).reshape(-1)
    assert np.abs(w - ref[None, :, None]).max() < 32 * 2.0 ** -53 * np.abs(ref).max()


def _units(bp, N, xe, u, w, kappa=None):
    """Largest error of an entry of w in units of 2^-53 (|A| |u|)_i."""
    el = Element(bp, N, xe, kappa)
    err, scale = np.abs(w - el(u)), el(u, magnitudes=True)
    assert not err[scale == 0].any()
    return float((err[scale > 0] / scale[scale > 0]).max()) * 2.0 ** 53


def _bound(N):
    """About 2 p1 + 12 roundings meet on a path through the FP64 form; the 1D tables and the factors of the
    library and of the reference differ by their own roundings, which the distances of neighbouring
    nodes amplify (1 / 0.13 at N = 7)."""
    return 4 * (N + 1) + 64


def _peak(N, bits, seed):
    """One corner value of 1, the others 2^-(bits+1) to 2^-bits with random signs."""
    r = uniform_pm1(seed, np.arange((N + 1) ** 3))
    u = np.ldexp(np.copysign(0.5 + 0.5 * np.abs(r), r), -bits)
    u[0] = 1.0
    return u


@pytest.mark.parametrize("bp,N", [(5, 1), (5, 3), (5, 4), (5, 7), (6, 3)])
@pytest.mark.parametrize("contrast", [1.0, 100.0, 1e5])
def test_coefficient_spread(bp, N, contrast):
    """kappa larger at the corner point where u is: the other entries of A u come from small values and
    small factors alone. (On a grid of the largest factor and value, 2^-60 of the product of both ratios
    was about 600 units at contrast 100.)"""
    op = pkg.Operator.box(bp, 2, 1, 1, N)
    kappa = np.ones((2, op.nquad ** 3))
    kappa[:, 0] = contrast
    op.set_kappa(torch.from_numpy(kappa).cuda())
    u = np.repeat(_peak(N, 3 if contrast == 1.0 else 6, 10)[None], 2, 0)
    w = _run(op, u if op.ncomp == 1 else np.repeat(u[..., None], 3, -1)).reshape(u.shape + (-1,))
    for e in range(2):
        assert _units(bp, N, op.coords[e], u[e], w[e, :, -1], kappa[e]) < _bound(N)


def _uneven(kind, N, seed):
    p1 = N + 1
    k, j, i = np.meshgrid(*[np.arange(p1)] * 3, indexing="ij")
    if kind.startswith("peak"):
        return _peak(N, int(kind[4:]), seed)
    if kind == "inner":  # the peak inside, on the longest list of neighbours
        u = _peak(N, 24, seed)
        u[0], u[u.size // 2] = u[1], 1.0
        return u
    if kind == "decay":
        return np.ldexp(1.0 - 0.25 * uniform_pm1(seed, np.arange(p1 ** 3)), -3 * (i + j + k).reshape(-1))
    if kind == "unit":
        u = np.zeros(p1 ** 3)
        u[p1 ** 3 // 3] = 1.0
        return u
    if kind == "plane":  # one large plane of nodes: every line across it is large, those along it are not
        return np.where(j == p1 - 1, 1.0, 2.0 ** -30).reshape(-1) * uniform_pm1(seed, np.arange(p1 ** 3))
    return uniform_pm1(seed, np.arange(p1 ** 3))


@pytest.mark.parametrize("bp,N", [(5, 1), (5, 2), (5, 4), (5, 5), (5, 7), (6, 3), (1, 1), (1, 3), (2, 3), (3, 1), (3, 2), (3, 5),
                                  (3, 7), (4, 3)])
@pytest.mark.parametrize("kind", ["random", "peak4", "peak12", "peak40", "inner", "decay", "unit", "plane"])
def test_uneven_values(bp, N, kind):
    """Every entry of A u to within a few units of 2^-53 (|A| |u|)_i, however the values of the element are spread."""
    op = pkg.Operator.box(bp, 3, 1, 1, N)
    u = np.stack([_uneven(kind, N, 11), uniform_pm1(12, np.arange((N + 1) ** 3)), _uneven(kind, N, 13)])
    u[2] = np.ldexp(u[2], -40)
    w = _run(op, u if op.ncomp == 1 else np.stack([u, u[::-1], u], -1)).reshape(u.shape + (-1,))
    for e in range(3):
        assert _units(bp, N, op.coords[e], u[e], w[e, :, -1]) < _bound(N)


@pytest.mark.parametrize("bp,N", [(5, 3), (5, 7), (5, 11), (3, 4), (6, 5)])
def test_uneven_values_beside_the_boundary(bp, N):
    """Rows of A u next to Dirichlet faces, edges and corners, where whole lines are masked to zero."""
    op = pkg.Operator.box(bp, 2, 2, 2, N)
    coords, l2g, dirichlet = pkg.mesh_box(2, 2, 2, N, 0.05)
    n = dirichlet.shape[0]
    for drop in (0, 30):
        u = uniform_pm1(14, np.arange(n))
        u = np.where(np.arange(n) % 3 == 0, u, np.ldexp(u, -drop)) * (1 - dirichlet)
        w = op.apply(torch.from_numpy(u if op.ncomp == 1 else np.stack([u] * 3, -1)).cuda()).cpu().numpy().reshape(n, -1)[:, -1]
        ref, scale = np.zeros(n, np.longdouble), np.zeros(n, np.longdouble)
        for e in range(8):
            el = Element(bp, N, coords[e])
            np.add.at(ref, l2g[e], el(u[l2g[e]]))
            np.add.at(scale, l2g[e], el(u[l2g[e]], magnitudes=True))
        free = dirichlet == 0
        assert np.abs(w[free] - ref[free]).max() < 1.0
        units = float((np.abs(w[free] - ref[free]) / scale[free]).max()) * 2.0 ** 53
        assert units < _bound(min(N, 7)) * (4 if N > 7 else 1)


@pytest.mark.parametrize("bp,N,E", [(3, 1, 15), (3, 2, 9), (3, 3, 6), (3, 5, 8), (3, 7, 3), (3, 12, 1), (4, 1, 29), (4, 4, 6),
                                    (4, 6, 2)])
@pytest.mark.parametrize("beta", [3.0, 1e6])
def test_helmholtz_is_the_sum_of_two_operators(bp, N, E, beta):
    """A u + beta B u of BP3/BP4 to two roundings of the sum of BP3's A u and beta times BP1's B u, block
    remainders and an uneven element included."""
    coords, l2g, _ = pkg.mesh_box(E, 1, 1, N, 0.05)
    stiff, mass = pkg.Operator(bp, N, coords, l2g, None), pkg.Operator(1 if bp == 3 else 2, N, coords, l2g, None)
    shape = (E, (N + 1) ** 3) if bp == 3 else (E, (N + 1) ** 3, 3)
    u = uniform_pm1(15, np.arange(int(np.prod(shape)))).reshape(shape)
    u[E // 2].reshape(-1)[1:] *= 1e-9
    a, b = _run(stiff, u), _run(mass, u)
    stiff.set_helmholtz(beta)
    assert (np.abs(_run(stiff, u) - (a + beta * b)) <= 2.0 ** -52 * (np.abs(a) + 2 * beta * np.abs(b))).all()


@pytest.mark.parametrize("bp,N", [(1, 1), (1, 4), (3, 2), (3, 7)])
def test_unassembled_pairs_are_the_fp64_results(bp, N):
    """Element-local vectors are FP64 on both sides: pair contexts of BP1/BP3 give the FP64 operator's bits."""
    u = uniform_pm1(16, np.arange(5 * (N + 1) ** 3)).reshape(5, -1)
    w = [_run(pkg.Operator.box(bp, 5, 1, 1, N, arith=arith), u) for arith in (pkg.ARITH_FP64, pkg.ARITH_DF64)]
    np.testing.assert_array_equal(w[0], w[1])


def test_pair_conversion_of_special_values():
    """Pairs whose parts are zero, tiny or not finite through an apply of the pair arithmetic."""
    op = pkg.Operator.box(1, 2, 1, 1, 2, arith=pkg.ARITH_DF64)
    ref = pkg.Operator.box(1, 2, 1, 1, 2)
    u = uniform_pm1(17, np.arange(op.nglobal))
    u[::3] = 0.0
    u[1::3] = np.ldexp(np.round(np.ldexp(u[1::3], 10)), -10)  # low parts zero
    t = torch.from_numpy(u).cuda()
    w, r = op.apply(t).cpu().numpy(), ref.apply(t).cpu().numpy()
    assert np.abs(w - r).max() < 2.0 ** -44 * np.abs(r).max()
    b = torch.from_numpy(r).cuda()
    x, info = op.solve(b, tol=1e-12)
    assert info["status"] == "OK" and float((x - t).abs().max()) < 1e-10
    b[3] = float("inf")
    with pytest.raises(pkg.CeedbpError):
        op.solve(b, tol=1e-12)


def _graded(N, ratio):
    """A box of one row of two elements whose nodes crowd towards x = y = z = 0: det J varies over more than
    `ratio` within each element."""
    coords, l2g, _ = pkg.mesh_box(2, 1, 1, N, 0.0)
    a = ratio ** (1.0 / 3.0)
    grade = lambda x: (x + 0.5 * (a - 1.0) * x * x) / (1.0 + 0.5 * (a - 1.0))
    out = coords.copy()
    out[0, :, 0], out[1, :, 0] = 0.5 * grade(2.0 * coords[0, :, 0]), 0.5 + 0.5 * grade(2.0 * coords[1, :, 0] - 1.0)
    out[..., 1], out[..., 2] = grade(coords[..., 1]), grade(coords[..., 2])
    return out, l2g


@pytest.mark.parametrize("bp,N", [(1, 2), (1, 5), (2, 3), (3, 3), (3, 7), (4, 4), (5, 5), (6, 2)])
@pytest.mark.parametrize("ratio", [8.0, 1e3, 1e5])
def test_factors_that_vary_within_an_element(bp, N, ratio):
    """Mass and stiffness factors on the grid and off it (spreads beyond 2^5), in every kernel."""
    coords, l2g = _graded(N, ratio)
    op = pkg.Operator(bp, N, coords, l2g, None)
    shape = (2, (N + 1) ** 3) if op.ncomp == 1 else (2, (N + 1) ** 3, 3)
    u = uniform_pm1(18, np.arange(int(np.prod(shape)))).reshape(shape)
    which = "B" if bp in (1, 2) else "A"
    w = _run(op, u)
    for e in range(2):
        ref = element_matrices(coords[e], N, bp_rule(bp, N), want=(which,))[which] @ u[e]
        assert np.linalg.norm(w[e] - ref) < 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("bp,N", [(3, 2), (3, 6), (4, 3)])
@pytest.mark.parametrize("contrast", [1e4, 0.0])
def test_coefficient_jumps_gauss(bp, N, contrast):
    """kappa jumping between the quadrature points of one element among others, also to zero."""
    op = pkg.Operator.box(bp, 3, 1, 1, N)
    kappa = np.ones((3, op.nquad ** 3))
    kappa[1, ::3] = contrast
    op.set_kappa(torch.from_numpy(kappa).cuda())
    shape = (3, (N + 1) ** 3) if op.ncomp == 1 else (3, (N + 1) ** 3, 3)
    u = uniform_pm1(19, np.arange(int(np.prod(shape)))).reshape(shape)
    w = _run(op, u)
    for e in range(3):
        ref = element_matrices(op.coords[e], N, bp_rule(bp, N), kappa=kappa[e], want=("A",))["A"] @ u[e]
        assert np.linalg.norm(w[e] - ref) < 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("bp,N,dims", [(1, 7, (4, 3, 3)), (1, 15, (2, 2, 2)), (2, 9, (2, 2, 1)), (3, 11, (2, 2, 2)), (5, 7, (4, 4, 4)),
                                       (5, 15, (2, 2, 2)), (6, 9, (2, 2, 2))])
@pytest.mark.parametrize("weighted", [True, False])
def test_solves_reach_the_residual_of_fp64(bp, N, dims, weighted):
    """CG takes uneven directions on the grid the later the further the residual has fallen: the same iteration
    counts and the same true residual as with every element in FP64, for right-hand sides B f and for values that
    span the quadrature weights from the first direction on."""
    op = pkg.Operator.box(bp, *dims, N)
    _, _, d = pkg.mesh_box(*dims, N)
    f = torch.from_numpy(uniform_pm1(23, np.arange(op.nglobal * op.ncomp)).reshape(tuple(op.empty().shape))).cuda()
    b = op.mass(f) if weighted else f
    if bp > 2:
        free = torch.from_numpy(1.0 - d).cuda()
        b = b * (free[:, None] if op.ncomp == 3 else free)
    out = []
    for on in (False, True):
        op.set_fixed_point(on)
        x, info = op.solve(b, tol=1e-12)
        op.set_fixed_point(False)
        out.append((info["iters"], float((b - op.apply(x)).norm() / b.norm())))
    assert all(abs(i - j) <= 1 for i, j in zip(out[0][0], out[1][0]))
    assert out[1][1] < 2.0 * out[0][1] + 1e-12
