"""Where node results go: written by the kernel into device arrays, packed and
copied once to host arrays, copied array by array when large or unaligned; any
mix of host and device arguments gives the same values."""
from __future__ import annotations

import ctypes

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

DEV = torch.device("cuda:0")


def nodes(t, k, seed):
    rng = np.random.default_rng(seed)
    lo = rng.uniform(-2, 1, (k, t.n_vars))
    return np.stack([lo, lo + rng.uniform(0.1, 1.0, lo.shape)], -1), rng.integers(1, 4, (k, t.n_vars)).astype(np.int32)


@pytest.mark.parametrize("k", [1, 37, 20000])          # 20000 nodes: more than the pinned staging takes
@pytest.mark.parametrize("host", [0b00000, 0b11111, 0b10101, 0b01010])
@pytest.mark.parametrize("batched", [1, 0])
def test_any_mix_of_host_and_device_results(k, host, batched):
    if not batched and k > 100:
        pytest.skip("one launch per node")
    t = W.random_problem(2, 30, 3, W.OPS_RATIONAL, [[-2, 2]] * 2, 9, "routing")
    boxes, splits = nodes(t, k, k)
    with ivb.Problem(t, max_nodes=max(k, 64)) as p:
        ref = p.bound_nodes_ex(boxes, splits, want_hull=True)
    with ivb.Problem(t, max_nodes=max(k, 64), batched=batched) as p:
        bd, sd = torch.from_numpy(boxes).to(DEV), torch.from_numpy(splits).to(DEV)
        want = [("lb", (k,)), ("infeasible", (k,)), ("ub", (k,)), ("minlo", (k, t.n_out)), ("maxhi", (k, t.n_out))]
        for rep in range(2):
            out, ptr, raw = [], [], []
            for i, (name, shape) in enumerate(want):
                dt = np.uint8 if name == "infeasible" else np.float64
                if host >> i & 1:
                    a = np.full(shape, 7, dt)
                    out.append(a)
                    ptr.append(a.ctypes.data)
                    raw.append(None)
                else:       # the second time the double arrays start 4 bytes off their alignment
                    off = 4 * rep
                    nb = int(np.prod(shape)) * np.dtype(dt).itemsize
                    r = torch.full((nb + 16,), 7, dtype=torch.uint8, device=DEV)
                    out.append((off, nb, shape, dt))
                    ptr.append(r.data_ptr() + off)
                    raw.append(r)
            b, s = (bd.data_ptr(), sd.data_ptr()) if rep else (boxes.ctypes.data, splits.ctypes.data)
            vp = ctypes.c_void_p
            st = ivb.lib().ivb_bound_nodes_ex(p._h, k, vp(b), vp(s), *(vp(x) for x in ptr), None)
            assert st == 0, p.ivb_last_error()
            torch.cuda.synchronize()
            for (name, _), o, r in zip(want, out, raw):
                v = o if r is None else r.cpu().numpy()[o[0]:o[0] + o[1]].tobytes()
                v = v if r is None else np.frombuffer(v, o[3]).reshape(o[2])
                assert np.array_equal(v, np.asarray(ref[name])), name
