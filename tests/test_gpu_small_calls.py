"""Calls of few subdomains share each subdomain's outputs among 2 or 4 threads of
the segmented kernel, or warp groups of the interpreter: the same bits as the
interpreter with one thread each on both sides of every switch, with constraints, the feasibility filter and calls of changing size on
one handle."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2507_20769_gb300 import build as B  # noqa: E402

B.build()
from paper_2507_20769_gb300 import ivb  # noqa: E402
from paper_2507_20769_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("n_ineq,filt,use_graph", [(0, 0, 1), (1, 1, 1), (3, 1, 0), (5, 0, 1)])
@pytest.mark.parametrize("specialize,form", [(3, "mvf"), (0, "mvf"), (0, "nie")])
def test_thread_count_follows_the_size_of_the_call(n_ineq, filt, use_graph, specialize, form):
    t = W.random_problem(2, 60, n_ineq, W.OPS_ALL, [[-2, 2]] * 2, 40 + n_ineq, "small calls")
    threads = 1024 * torch.cuda.get_device_properties(0).multi_processor_count
    with ivb.Problem(t, specialize=specialize, form=form, filter=filt, use_graph=use_graph, autotune=0) as p, \
            ivb.Problem(t, specialize=0, form=form, filter=filt, autotune=0, threads_per_subdomain=1) as q:
        for total in (1, 33, threads // 4, threads // 4 + 1, threads // 2, threads // 2 + 1, threads + 1, 7):
            a = max(1, total // 3)
            boxes = np.array([[[-2.0, 0.5], [-1.0, 2.0]], [[0.5, 2.0], [-2.0, 0.25]]])
            splits = np.array([[a, 1], [max(1, total - a), 1]], np.int32)
            r = p.bound_nodes_ex(boxes, splits, want_hull=True)
            ref = q.bound_nodes_ex(boxes, splits, want_hull=True)
            for k in ("lb", "ub", "minlo", "maxhi", "infeasible"):
                assert np.array_equal(r[k].view(np.uint8), ref[k].view(np.uint8)), (total, k)
