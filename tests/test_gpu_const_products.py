"""Products by constants in the segmented kernel (powers of two as exponent
steps, other constants with their sign known): node hulls bit for bit the
oracle's and bytewise the interpreter's, with zero ends, subnormal, huge and
overflowing operands, constants of either sign and magnitude, and first and
later contributions to an adjoint."""
from __future__ import annotations

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2507_20769_gb300 import build as B  # noqa: E402

B.build()
from paper_2507_20769_gb300 import ivb  # noqa: E402
from paper_2507_20769_gb300.workloads import KIND_INEQ, KIND_OBJ  # noqa: E402
import problems as P  # noqa: E402

CONSTANTS = [1.0, -1.0, 0.5, -2.0, 2.0 ** -30, -2.0 ** 200, 2.0 ** 999, -2.0 ** -999, 2.0 ** 1010, 2.0 ** -1060,
             3.7, -1.0 / 3.0, 1.0e-300, -1.7e308, 0.0, -0.0]


@pytest.mark.parametrize("form", ["mvf", "nie"])
def test_constant_factors(form):
    Bd = P.Builder(2)
    for k, c in enumerate(CONSTANTS):
        x, y, cc = Bd.x(0), Bd.x(1), Bd.const(c)
        a = Bd.mul(x, cc)                       # constant on the right
        b = Bd.mul(cc, Bd.mul(x, y))            # constant on the left
        s = Bd.sub(Bd.mul(a, y), Bd.add(a, b))  # a read twice: first and later contributions
        Bd.output(s, KIND_OBJ if k == 0 else KIND_INEQ)
    t = Bd.tape([[-1.0, 1.0], [-1.0, 1.0]], "constant factors")
    boxes = np.array([[[-1.0, 1.0], [-2.0, 3.0]], [[0.0, 2.0], [-0.0, 0.0]], [[-3e-308, 2e-308], [0.25, 4.0]],
                      [[1.0e300, 1.01e300], [-1.0, 1.0]], [[-1.0e300, -1.0e290], [1e-300, 7.0]], [[0.3, 0.3], [-5.0, -0.0]]])
    splits = np.array([[8, 6], [4, 1], [5, 3], [3, 4], [2, 2], [1, 7]], np.int32)
    ref = oracle.bound_nodes(t, boxes, splits, grad_mode="adjoint", form=form, tight=True)
    with ivb.Problem(t, form=form) as p:
        ri = p.bound_nodes_ex(boxes, splits, want_hull=True)
    with ivb.Problem(t, form=form, specialize=3, seg_chunk=16) as p:
        rs = p.bound_nodes_ex(boxes, splits, want_hull=True)
    for k in ("lb", "ub", "minlo", "maxhi"):
        assert np.array_equal(ri[k], ref[k]), k
        assert np.array_equal(rs[k].view(np.int64), ri[k].view(np.int64)), k
