"""The arithmetic of an operator does not depend on what else is allocated at setup, fixed-point factors make
room for later calls, and operators without them work in FP64."""
import numpy as np
import pytest
import torch

import paper_2004_06722_gb300 as pkg
from oracle.problems import BakeoffProblem
from synth import uniform_pm1

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    pkg.load_library()


DIMS, N = (32, 32, 32), 7  # 0.8 GB of fixed-point factors
FX_BYTES = 48 * 32 ** 3 * 512


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.fixture(scope="module")
def mesh():
    return pkg.mesh_box(*DIMS, N, 0.05)


@pytest.fixture(scope="module")
def reference(mesh):
    """(values, A u, bytes of the operator without fixed-point factors)"""
    u = torch.from_numpy(uniform_pm1(1, np.arange(mesh[2].shape[0]))).cuda()
    op = pkg.Operator(5, N, *mesh)
    w = op.apply(u).clone()
    op.close()
    before = _free()
    op = pkg.Operator(5, N, *mesh)
    after = _free()
    op.close()
    return u, w, before - after - FX_BYTES


def _fill(leave):
    """All but `leave` bytes of the device's free memory."""
    torch.cuda.empty_cache()
    hold = torch.empty(_free() - int(leave), dtype=torch.uint8, device="cuda")
    return hold


def test_same_bits_when_little_memory_is_free(mesh, reference):
    u, w, base = reference
    hold = _fill(base + 2 * FX_BYTES)  # the factors are half of what is free when they are made
    try:
        op = pkg.Operator(5, N, *mesh)
        same = torch.equal(op.apply(u, torch.empty_like(w)), w)
        op.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert same


def test_setup_without_room_for_the_factors(mesh, reference):
    u, w, base = reference
    hold = _fill(base + 0.85 * FX_BYTES)
    try:
        op = pkg.Operator(5, N, *mesh)
        on, left = op.fixed_point, _free()
        x = op.apply(u, torch.empty_like(w))
        op.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert not on and left > 0.75 * FX_BYTES  # nothing of them stays allocated
    assert float((x - w).norm()) < 1e-13 * float(w.norm())


def test_factors_make_room_for_set_kappa(mesh, reference):
    u, w, base = reference
    kappa = torch.full((DIMS[0] * DIMS[1] * DIMS[2], (N + 1) ** 3), 2.0, dtype=torch.float64, device="cuda")
    hold = _fill(base + 1.6 * FX_BYTES)
    try:
        op = pkg.Operator(5, N, *mesh)
        first = op.fixed_point
        op.set_kappa(kappa)  # keeps the factors without kappa: as large as the fixed-point ones
        then, x = op.fixed_point, op.apply(u, torch.empty_like(w))
        op.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert first and not then
    assert float((x - 2.0 * w).norm()) < 1e-13 * float(w.norm())


@pytest.mark.parametrize("bp,order,arith", [(1, 1, 0), (1, 7, 0), (2, 3, 0), (3, 1, 0), (3, 4, 0), (3, 8, 0), (4, 2, 0), (4, 6, 0),
                                            (5, 1, 0), (5, 4, 0), (5, 7, 0), (5, 10, 0), (6, 2, 0), (6, 7, 0), (1, 5, 1),
                                            (3, 6, 1), (3, 15, 0), (5, 15, 0), (6, 14, 0)])
def test_without_fixed_point_factors(bp, order, arith):
    """Apply, unassembled apply and solve in FP64 against the oracle, and the first bits again with the factors back."""
    dims = (3, 2, 2) if order < 8 else (2, 1, 1)
    ref = BakeoffProblem(bp, *dims, order, amp=0.05)
    op = pkg.Operator.box(bp, *dims, order, arith=arith)
    shape = tuple(op.empty().shape)
    uh = uniform_pm1(2, np.arange(int(np.prod(shape)))).reshape(shape)
    u = torch.from_numpy(uh).cuda()
    first = op.apply(u)
    assert op.fixed_point
    op.set_fixed_point(False)
    assert not op.fixed_point
    w = op.apply(u)
    w_ref = ref.apply(uh)
    assert np.linalg.norm(w.cpu().numpy() - w_ref) < 1e-12 * np.linalg.norm(w_ref)
    b = ref.rhs(uh)
    x, info = op.solve(torch.from_numpy(b).cuda(), tol=1e-8)
    assert info["status"] == "OK"
    op.set_fixed_point(True)
    x2, info2 = op.solve(torch.from_numpy(b).cuda(), tol=1e-8)
    assert all(abs(p - q) <= 1 for p, q in zip(info["iters"], info2["iters"]))
    assert op.fixed_point and torch.equal(op.apply(u), first)


def test_fixed_point_belongs_to_some_contexts():
    for kw in (dict(arith=pkg.ARITH_DF64), dict(geom=pkg.GEOM_RECOMPUTE)):
        op = pkg.Operator.box(5, 2, 2, 2, 3, **kw)
        assert not op.fixed_point
        with pytest.raises(pkg.CeedbpError) as err:
            op.set_fixed_point(True)
        assert err.value.status == pkg.EUNSUPPORTED
