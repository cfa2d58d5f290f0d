"""The direct-stiffness sums on local-to-global maps that no box mesh has: nodes shared by 1 to 13 elements, nodes
that no element touches, and the longest list last (where the gather reads into the padding)."""
import numpy as np
import pytest
import torch

import paper_2004_06722_gb300 as pkg
from synth import uniform_pm1

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    pkg.load_library()


E, N = 13, 2


def _mesh():
    """13 separate unit elements; local node a of element e is shared by a group of elements, the same local
    node of each. Valences 1..13, 7 unused nodes, the node of valence 13 is the last one."""
    coords, _, _ = pkg.mesh_box(1, 1, 1, N, 0.05)
    p3 = (N + 1) ** 3
    l2g = np.empty((E, p3), np.int64)
    nxt = 7  # nodes 0..6 belong to nobody
    for a in range(p3):
        if a == p3 - 1:
            break
        size, e = a % 13 + 1, 0
        while e < E:
            k = min(size, E - e)
            l2g[e:e + k, a] = nxt
            nxt, e = nxt + 1, e + k
    l2g[:, p3 - 1] = nxt
    return np.repeat(coords, E, 0), l2g, nxt + 1


def _gathered(op, l2g, n, u):
    """Q^T A_L Q u with the library's element kernel and a sum over slots in ascending order."""
    uL = torch.from_numpy(u[l2g]).cuda()
    wL = op.bk_apply(uL).cpu().numpy()
    w = np.zeros_like(u)
    for e in range(E):
        np.add.at(w, l2g[e], wL[e])
    return w


@pytest.mark.parametrize("bp,arith", [(1, 0), (2, 0), (3, 0), (4, 0), (5, 0), (6, 0), (1, 1), (3, 1), (5, 1), (6, 1)])
def test_apply_on_any_valence(bp, arith):
    coords, l2g, n = _mesh()
    op = pkg.Operator(bp, N, coords, l2g, np.zeros(n, np.uint8), arith=arith)
    u = uniform_pm1(20, np.arange(n * op.ncomp)).reshape((n,) if op.ncomp == 1 else (n, 3))
    w, ref = op.apply(torch.from_numpy(u).cuda()).cpu().numpy(), _gathered(op, l2g, n, u)
    assert not w[:7].any()
    if arith == 0:
        np.testing.assert_array_equal(w, ref)
    else:
        assert np.abs(w - ref).max() < 2.0 ** -40 * np.abs(ref).max()


def _cg(apply, dinv, b, iters):
    x, r = np.zeros_like(b), b.copy()
    p = z = dinv * r
    for _ in range(iters):
        w = apply(p)
        rz = float(r @ z)
        a = rz / float(p @ w)
        x, r = x + a * p, r - a * w
        z = dinv * r
        p = z + float(r @ z) / rz * p
    return x


@pytest.mark.parametrize("bp,arith", [(1, 0), (5, 0), (1, 1), (5, 1)])
def test_cg_iterations_on_any_valence(bp, arith):
    """Two iterations against the textbook recurrence; BP5 with the nodes of valence 2 held as boundary."""
    coords, l2g, n = _mesh()
    valence = np.bincount(l2g.reshape(-1), minlength=n)
    d = (valence == 2).astype(np.uint8) if bp == 5 else np.zeros(n, np.uint8)
    op = pkg.Operator(bp, N, coords, l2g, d, arith=arith)
    free = (d == 0) & (valence > 0)
    b = uniform_pm1(21, np.arange(n)) * free
    dinv = op.jacobi().cpu().numpy()
    x, _ = op.solve(torch.from_numpy(b).cuda(), fixed_iters=2)
    ref = _cg(lambda p: _gathered(op, l2g, n, p * free) * free, np.where(free, dinv, 0.0), b, 2)
    assert np.linalg.norm(x.cpu().numpy() - ref) < 1e-11 * np.linalg.norm(ref)


def test_mixed_and_batch_on_any_valence():
    """The FP32 inner iteration and batched solves (FP64 and pairs) against the single FP64 solve."""
    coords, l2g, n = _mesh()
    valence = np.bincount(l2g.reshape(-1), minlength=n)
    d = ((valence == 2) | (valence == 0)).astype(np.uint8)
    op = pkg.Operator(5, N, coords, l2g, d)
    b = torch.from_numpy(uniform_pm1(22, np.arange(n)) * (1 - d)).cuda()
    x, _ = op.solve(b, tol=1e-11)
    op.prepare_mixed(pkg.MIXED_FP32)
    y, _ = op.solve(b, tol=1e-11, mixed=pkg.MIXED_FP32)
    assert float((y - x).norm()) < 1e-8 * float(x.norm())
    for arith in (pkg.ARITH_FP64, pkg.ARITH_DF64):
        batch = pkg.Batch([(N, coords, l2g, d)] * 2, arith=arith)
        xs, _ = batch.solve([b, 2.0 * b], tol=1e-11)
        assert float((xs[0] - x).norm()) < 1e-8 * float(x.norm())
        assert float((xs[1] - 2.0 * x).norm()) < 2e-8 * float(x.norm())
        batch.close()
