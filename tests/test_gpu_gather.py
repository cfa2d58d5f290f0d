"""The direct-stiffness sums of the vector kernels around the sizes where the grid (1216 blocks of 256)
holds every node once or twice: one node in flight per thread up to there, two above.

Tolerances. A sum has at most 8 terms, in an order of its own on each side: 2 * 7 roundings of 2^-53 of
the sum of their magnitudes, 2e-15. Two iterations of CG: scalars from sums over 6e5 nodes, whose tree of
partial sums is at most ~30 deep on either side (4e-15 each), enter through two quotients and two
recurrences each: 1e-12 leaves a factor of ten."""
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


# nodes of order 1: 8; 311296 = 1216 * 256; 4096 more; twice as many; 9728 more
@pytest.mark.parametrize("bp", [5, 6])
@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 3, 2), (63, 63, 75), (63, 63, 76), (63, 127, 75), (64, 127, 75)])
def test_sums_and_update(bp, dims):
    coords, l2g, dirichlet = pkg.mesh_box(*dims, 1, 0.05)
    op = pkg.Operator(bp, 1, coords, l2g, dirichlet)
    n, nc = op.nglobal, op.ncomp
    shape = (n,) if nc == 1 else (n, nc)
    u = torch.from_numpy(uniform_pm1(9, np.arange(n * nc)).reshape(shape)).cuda()
    mask = torch.from_numpy(1.0 - dirichlet.astype(np.float64)).cuda().reshape((n,) + (1,) * (nc > 1))
    u *= mask
    idx = torch.from_numpy(l2g.reshape(-1)).cuda()
    wl = op.bk_apply(u[idx].reshape((l2g.shape[0], 8) + shape[1:])).reshape((-1,) + shape[1:])
    w = torch.zeros_like(u).index_add_(0, idx, wl) * mask
    mag = torch.zeros_like(u).index_add_(0, idx, wl.abs())
    assert bool(((op.apply(u) - w).abs() <= 2e-15 * mag).all())

    if dims == (1, 1, 1):  # no interior node
        return
    x, info = op.solve(u, fixed_iters=2)
    dinv = op.jacobi().reshape(mask.shape)
    cols = [slice(None)] if nc == 1 else [(slice(None), c) for c in range(nc)]
    xr, r, p, rz = torch.zeros_like(u), u.clone(), dinv * u, [0.0] * nc
    for c, k in enumerate(cols):
        rz[c] = (r[k] * p[k]).sum()
    for _ in range(2):
        q = op.apply(p)
        for c, k in enumerate(cols):
            a = rz[c] / (p[k] * q[k]).sum()
            xr[k] += a * p[k]
            r[k] -= a * q[k]
            z = dinv.reshape(-1) * r[k]
            new = (r[k] * z).sum()
            p[k] = z + new / rz[c] * p[k]
            rz[c] = new
    assert float((x - xr).abs().max()) < 1e-12 * float(xr.abs().max())
