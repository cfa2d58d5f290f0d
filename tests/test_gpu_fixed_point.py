"""The block fixed-point FP64 element kernels: accuracy at every order, sequence and block remainders,
and the values that do not fit an element's grid (they run in FP64 inside the same kernel).

Tolerances: one application against the oracle 1e-12 (the bar of the FP64 path); scaling by a power of
two is exact in exact arithmetic and in the grid's (1e-13 covers the FP64 form's different rounding).
"""
import numpy as np
import pytest
import torch

import paper_2004_06722_gb300 as pkg
from oracle.element import element_matrices
from oracle.mesh import box_mesh
from oracle.quadrature import bp_rule
from synth import uniform_pm1

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    pkg.load_library()


def _local(bp, dims, N, uL, kappa=None):
    coords, _ = box_mesh(*dims, N, 0.05)
    rule = bp_rule(bp, N)
    which = "B" if bp in (1, 2) else "A"
    out = np.zeros_like(uL)
    for e in range(coords.shape[0]):
        kw = {} if kappa is None else {"kappa": kappa[e]}
        out[e] = element_matrices(coords[e], N, rule, want=(which,), **kw)[which] @ uL[e]
    return out


def _run(op, uL):
    return op.bk_apply(torch.from_numpy(uL).cuda()).cpu().numpy()


# element counts around the elements per block (32, 14, 8, 5, 7 and 1 from order 1 up)
CASES = [(5, 1, 31), (5, 1, 33), (5, 2, 15), (5, 3, 9), (5, 4, 6), (5, 5, 8), (5, 6, 3), (5, 8, 2), (5, 9, 2),
         (5, 10, 1), (5, 11, 1), (5, 12, 1), (6, 1, 33), (6, 4, 6), (6, 6, 2), (6, 9, 1),
         (1, 1, 15), (1, 2, 9), (1, 3, 4), (1, 4, 8), (1, 5, 2), (1, 8, 2), (1, 12, 1), (2, 2, 9), (2, 6, 2), (2, 11, 1),
         (3, 1, 15), (3, 2, 7), (3, 3, 6), (3, 4, 6), (3, 6, 3), (3, 8, 2), (3, 10, 1), (3, 11, 1), (3, 12, 1),
         (4, 1, 15), (4, 3, 6), (4, 5, 2), (4, 9, 1)]


@pytest.mark.parametrize("bp,N,E", CASES)
def test_element_operator(bp, N, E):
    op = pkg.Operator.box(bp, E, 1, 1, N)
    p3 = (N + 1) ** 3
    shape = (E, p3) if op.ncomp == 1 else (E, p3, 3)
    uL = uniform_pm1(3, np.arange(int(np.prod(shape)))).reshape(shape)
    ref = _local(bp, (E, 1, 1), N, uL)
    w = _run(op, uL)
    assert np.linalg.norm(w - ref) < 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("bp,N", [(5, 2), (5, 3), (5, 7), (6, 5), (1, 3), (2, 2), (3, 4), (3, 7), (4, 3)])
def test_element_sequences_agree(bp, N):
    """Every copy of one element in a mesh long enough for element sequences gives the same bits."""
    E = 40000 if N < 6 else 9000
    coords, l2g, _ = pkg.mesh_box(1, 1, 1, N, 0.05)
    p3 = (N + 1) ** 3
    op = pkg.Operator(bp, N, np.repeat(coords, E, 0), np.arange(E * p3, dtype=np.int64).reshape(E, p3), None)
    one = uniform_pm1(4, np.arange(p3 * op.ncomp)).reshape((1, p3) if op.ncomp == 1 else (1, p3, 3))
    w = op.bk_apply(torch.from_numpy(np.repeat(one, E, 0)).cuda())
    assert bool((w == w[:1]).all())


@pytest.mark.parametrize("bp,N", [(5, 3), (5, 6), (5, 7), (5, 15), (1, 5), (3, 7), (3, 15), (4, 2)])
@pytest.mark.parametrize("k", [-900, -400, 300, 700])
def test_power_of_two_scaling(bp, N, k):
    """2^k u: inside the grid's exponent range the same integers, outside it the FP64 form."""
    op = pkg.Operator.box(bp, 2, 1, 1, N)
    shape = (2, (N + 1) ** 3) if op.ncomp == 1 else (2, (N + 1) ** 3, 3)
    uL = uniform_pm1(5, np.arange(int(np.prod(shape)))).reshape(shape)
    w0, w1 = _run(op, uL), np.ldexp(_run(op, np.ldexp(uL, k)), -k)
    if abs(k) <= 400:
        np.testing.assert_array_equal(w0, w1)
    else:
        assert np.linalg.norm(w1 - w0) < 1e-13 * np.linalg.norm(w0)


@pytest.mark.parametrize("N", [2, 5, 7])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_values(N, bad):
    """A non-finite node reaches exactly the nodes that share one of its coordinate planes, and no
    other element."""
    p1 = N + 1
    op = pkg.Operator.box(5, 1, 1, 3, N)
    uL = uniform_pm1(6, np.arange(3 * p1 ** 3)).reshape(3, -1)
    clean = _run(op, uL)
    a, b, c = 1, 0, p1 - 1
    uL[1, a + p1 * (b + p1 * c)] = bad
    w = _run(op, uL)
    k, j, i = np.meshgrid(*[np.arange(p1)] * 3, indexing="ij")
    hit = ((i == a) | (j == b) | (k == c)).reshape(-1)
    assert not np.isfinite(w[1][hit]).any() and np.isfinite(w[1][~hit]).all()
    assert np.abs(w[[0, 2]] - clean[[0, 2]]).max() < 1e-12 * np.abs(clean).max()


@pytest.mark.parametrize("bp,N", [(1, 3), (1, 7), (3, 4), (3, 7)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values_gauss(bp, N, bad):
    """Interpolation reaches every node of the element, and no other element."""
    op = pkg.Operator.box(bp, 1, 3, 1, N)
    uL = uniform_pm1(6, np.arange(3 * (N + 1) ** 3)).reshape(3, -1)
    clean = _run(op, uL)
    uL[1, 5] = bad
    w = _run(op, uL)
    assert not np.isfinite(w[1]).any()
    assert np.abs(w[[0, 2]] - clean[[0, 2]]).max() < 1e-12 * np.abs(clean).max()


@pytest.mark.parametrize("N,contrast", [(3, 30.0), (7, 100.0), (7, 1e6), (4, 1e9), (5, 0.0)])
def test_coefficient_contrast(N, contrast):
    """kappa jumping inside an element: below 2^7 on the grid, above it (and with zeros) in FP64."""
    op = pkg.Operator.box(5, 2, 2, 1, N)
    p3 = (N + 1) ** 3
    kappa = np.ones((4, p3))
    kappa[1, ::2] = contrast
    kappa[3] = 1e-3
    op.set_kappa(torch.from_numpy(kappa).cuda())
    uL = uniform_pm1(7, np.arange(4 * p3)).reshape(4, -1)
    ref = _local(5, (2, 2, 1), N, uL, kappa)
    w = _run(op, uL)
    for e in range(4):
        assert np.linalg.norm(w[e] - ref[e]) < 1e-12 * np.linalg.norm(ref[e])


@pytest.mark.parametrize("bp,N", [(5, 4), (6, 3), (1, 4), (3, 5)])
def test_zero_and_sparse_elements(bp, N):
    op = pkg.Operator.box(bp, 3, 1, 1, N)
    p3 = (N + 1) ** 3
    shape = (3, p3) if op.ncomp == 1 else (3, p3, 3)
    uL = np.zeros(shape)
    assert not _run(op, uL).any()
    uL[1, 7] = 1e-30
    w = _run(op, uL)
    ref = _local(bp, (3, 1, 1), N, uL)
    assert not w[0].any() and not w[2].any()
    assert np.linalg.norm(w - ref) < 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("N", [3, 4, 5, 6, 7, 8, 10, 11, 12])
@pytest.mark.parametrize("dims", [(6, 5, 5), (6, 6, 5)])
def test_threads_per_column(N, dims):
    """Three threads per column while every element has an SM of its own (152: 150 elements), one above
    (180): the first and the last elements against the oracle, on elements of even proportions."""
    E = dims[0] * dims[1] * dims[2]
    op = pkg.Operator.box(5, *dims, N)
    uL = uniform_pm1(8, np.arange(E * (N + 1) ** 3)).reshape(E, -1)
    w = _run(op, uL)
    rule = bp_rule(5, N)
    for e in (0, 1, E - 2, E - 1):
        ref = element_matrices(op.coords[e], N, rule, want=("A",))["A"] @ uL[e]
        assert np.linalg.norm(w[e] - ref) < 1e-12 * np.linalg.norm(ref)
