"""Values at the ends of FP64's range and of uneven magnitude in the block fixed-point element kernels."""
import numpy as np
import pytest
import torch

import paper_2004_06722_gb300 as pkg
from oracle.element import element_matrices
from oracle.quadrature import bp_rule
from synth import uniform_pm1

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
