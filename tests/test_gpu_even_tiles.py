"""Subdomain ranges dealt out evenly over the blocks: every subdomain is bounded
exactly once at the edges of warps, blocks and passes. One-variable cubic,
node hulls and stored enclosures bit for bit against the oracle."""
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
import problems as P  # noqa: E402

WAVE = 1024 * torch.cuda.get_device_properties(0).multi_processor_count
KEYS = ("lb", "ub", "minlo", "maxhi")


@pytest.mark.parametrize("specialize", [0, 1, 3])
def test_node_hulls_at_the_edges_of_passes(specialize):
    t = P.cubic_fig5()
    with ivb.Problem(t, specialize=specialize, autotune=0) as p:
        for total in (1, 31, 32, 33, 1023, 1025, WAVE - 1, WAVE, WAVE + 1, 2 * WAVE + 33, 5 * WAVE + 4097):
            # two nodes, the boundary between them inside a warp
            a = max(1, total // 3)
            splits = np.array([[a], [max(1, total - a)]], np.int32)
            boxes = np.array([[[-1.0, 0.7]], [[0.7, 2.0]]])
            r = p.bound_nodes_ex(boxes, splits, want_hull=True)
            ref = oracle.bound_nodes(t, boxes, splits, grad_mode="adjoint", tight=True)
            for k in KEYS:
                assert np.array_equal(r[k], ref[k]), (total, k)


@pytest.mark.parametrize("specialize", [0, 3])
def test_stored_ranges_at_the_edges_of_passes(specialize):
    t = P.cubic_fig5()
    box, splits = np.array([[-1.0, 2.0]]), np.array([3 * WAVE], np.int32)
    with ivb.Problem(t, specialize=specialize, autotune=0) as p:
        for first, count in ((0, 1), (5, 33), (WAVE - 7, 129), (77, WAVE + 1), (2 * WAVE + 1, WAVE - 1)):
            F, Fc, G = p.enclose(box, splits, first=first, count=count, want_fc=True, want_g=True)
            ref = oracle.enclose(t, box, splits, first=first, count=count, grad_mode="adjoint", tight=True,
                                 want_fc=True, want_g=True)
            for x, y in zip((F, Fc, G), ref):
                assert np.array_equal(x, y), (first, count)
