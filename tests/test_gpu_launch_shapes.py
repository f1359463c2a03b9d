"""Launch shapes fixed by options: the shape that runs is the documented one, and
the bounds are the interpreter's bits at every one of them."""
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

KEYS = ("lb", "ub", "minlo", "maxhi", "infeasible")


def tape():
    return W.random_problem(2, 60, 3, W.OPS_ALL, [[-2, 2]] * 2, 51, "launch shapes")


def bounds(p, total=7001):
    boxes = np.array([[[-2.0, 0.5], [-1.0, 2.0]], [[0.5, 2.0], [-2.0, 0.25]]])
    splits = np.array([[total // 3, 1], [total - total // 3, 1]], np.int32)
    return p.bound_nodes_ex(boxes, splits, want_hull=True)


def assert_same(r, ref, what):
    for k in KEYS:
        assert np.array_equal(r[k].view(np.uint8), ref[k].view(np.uint8)), (what, k)


@pytest.fixture(scope="module")
def reference():
    with ivb.Problem(tape(), specialize=0, autotune=0, threads_per_subdomain=1) as p:
        return bounds(p)


@pytest.mark.parametrize("sync", [0, 1])
@pytest.mark.parametrize("block,asked,runs", [(96, 2, 1), (96, 4, 1), (160, 2, 1), (192, 2, 2), (192, 4, 1), (32, 2, 1),
                                              (64, 2, 2), (128, 4, 4)])
def test_threads_per_subdomain_only_in_whole_warps(reference, block, asked, runs, sync):
    with ivb.Problem(tape(), specialize=3, seg_chunk=24, block_threads=block, threads_per_subdomain=asked,
                     seg_sync=sync) as p:
        r = bounds(p)
        tun = p.get_tuning()
    assert (tun["block_threads"], tun["threads_per_subdomain"]) == (block, runs)
    assert_same(r, reference, (block, asked))


def used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.mark.parametrize("specialize", [0, 3])
def test_stored_range_holds_frames_of_the_blocks_that_work(specialize):
    """a long tape (some 6 KB of frame per thread): one subdomain takes a block's frames, and a
    shape fixed by options bounds those of a range that fills the device; the same bits either way"""
    wl = W.config_workload(4)
    box, splits = wl.tape.root_box, np.asarray(wl.splits, np.int32)
    out = []
    for opts, ranges in ((dict(), ((77, 1),)), (dict(block_threads=32, blocks_per_sm=1), ((77, 1), (70, 40_000)))):
        with ivb.Problem(wl.tape, specialize=specialize, autotune=0, **opts) as p:
            warm = used()
            for first, count in ranges:
                out.append(p.enclose(box, splits, first=first, count=count, want_fc=True, want_g=True))
            assert used() - warm < 128 << 20
    for k in range(3):
        a, b, c = (np.asarray(o[k]) for o in out)
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
        assert np.array_equal(a.view(np.uint8), np.ascontiguousarray(c[7:8]).view(np.uint8))


@pytest.mark.parametrize("autotune", [0, 1])
def test_short_memory_runs_on_fewer_blocks(autotune):
    """frames that do not fit beside what the program holds: fewer blocks, the same bits"""
    t = W.config_tape(5)
    boxes = W.bisection_frontier(t.root_box, 64, seed=2026)[:1]
    splits = np.array([W.full_scale_splits(b, t.root_box) for b in boxes], np.int32)
    with ivb.Problem(t, specialize=0, autotune=0) as p:
        before = used()
        ref = p.bound_nodes_ex(boxes, splits, want_hull=True)
        full = used() - before
        F = p.enclose(boxes[0], splits[0], first=5, count=20_000)[0]
    assert full > 1 << 30
    with ivb.Problem(t, specialize=0, autotune=autotune) as p:
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        hog = torch.empty(free - full * 6 // 10, dtype=torch.uint8, device="cuda:0")
        try:
            for _ in range(2):
                assert_same(p.bound_nodes_ex(boxes, splits, want_hull=True), ref, "bounds")
            G = p.enclose(boxes[0], splits[0], first=5, count=20_000)[0]
        finally:
            del hog
            torch.cuda.empty_cache()
    assert np.array_equal(F.view(np.uint8), G.view(np.uint8))


@pytest.mark.parametrize("seg_regs", [64, 73, 82, 100, 128, 170, 255])
def test_every_register_budget_launches(reference, seg_regs):
    """the default block of a segmented kernel fits an SM whatever the budget"""
    with ivb.Problem(W.config_tape(2), specialize=3, autotune=0, seg_regs=seg_regs) as p:
        c2 = p.bound_nodes_ex(W.config_tape(2).root_box[None], np.full((1, 4), 5, np.int32), want_hull=True)
        assert p.get_tuning()["block_threads"] * -(-seg_regs // 8) * 8 <= 65536
    with ivb.Problem(W.config_tape(2), specialize=0, autotune=0) as p:
        assert_same(c2, p.bound_nodes_ex(W.config_tape(2).root_box[None], np.full((1, 4), 5, np.int32), want_hull=True),
                    seg_regs)
    with ivb.Problem(tape(), specialize=3, autotune=0, seg_regs=seg_regs) as p:
        assert_same(bounds(p), reference, seg_regs)


@pytest.mark.parametrize("specialize", [3, -1])
@pytest.mark.parametrize("block,per_sm,runs,regs", [(256, 0, 2, 128), (128, 0, 4, 128), (256, 2, 2, 128), (256, 4, 4, 64),
                                                    (0, 2, 1, 64)])
def test_fixed_shape_sets_the_register_budget(reference, specialize, block, per_sm, runs, regs):
    """configuration 2's chunks use most of their budget: the former shapes keep 128 registers"""
    t = W.config_tape(2)
    with ivb.Problem(t, specialize=specialize, autotune=0, block_threads=block, blocks_per_sm=per_sm) as p:
        r = p.bound_nodes_ex(t.root_box[None], np.full((1, 4), 5, np.int32), want_hull=True)
        tun, spec = p.get_tuning(), p.get_specialization()
    assert (tun["kernel"], tun["block_threads"], tun["blocks_per_sm"]) == (2, block or 1024, runs)
    assert regs - 16 < spec["registers"] <= regs
    with ivb.Problem(t, specialize=0, autotune=0) as p:
        assert_same(r, p.bound_nodes_ex(t.root_box[None], np.full((1, 4), 5, np.int32), want_hull=True), block)


@pytest.mark.parametrize("opts,which", [(dict(specialize=-1), 2), (dict(specialize=3), 2), (dict(specialize=1), 2),
                                        (dict(specialize=0), 2), (dict(specialize=-1), "small"),
                                        (dict(specialize=-1, grad_mode="forward"), 2)])
def test_the_tuned_shape_can_be_asked_for(opts, which):
    """what get_tuning reports goes back in as options: the same launch, the same bits"""
    t = W.config_tape(2) if which == 2 else W.random_problem(4, 14, 0, W.OPS_ALL, [[-2, 2]] * 4, 8, "small")
    boxes = W.bisection_frontier(t.root_box, 8, seed=20)
    splits = np.full((8, t.n_vars), 14, np.int32)
    with ivb.Problem(t, **opts) as p:
        ref = p.bound_nodes_ex(boxes, splits, want_hull=True)
        tun = p.get_tuning()
        assert tun["candidates"] > 0
    fixed = {k: tun[k] for k in ("block_threads", "blocks_per_sm", "tile", "frame_in_shared", "threads_per_subdomain")}
    with ivb.Problem(t, seg_sync=tun["chunk_sync"], **dict(opts, **fixed)) as p:
        r = p.bound_nodes_ex(boxes, splits, want_hull=True)
        again = p.get_tuning()
        if tun["kernel"] == 0 and p.get_specialization()["active"]:
            fixed.pop("frame_in_shared")   # the compiled kernel has none
    assert {k: again[k] for k in fixed} == {k: tun[k] for k in fixed}
    assert_same(r, ref, fixed)


@pytest.mark.parametrize("block", [288, 512, 672, 992, 1024])
def test_segmented_kernel_at_any_block(reference, block):
    with ivb.Problem(tape(), specialize=3, seg_chunk=24, block_threads=block) as p:
        assert_same(bounds(p), reference, block)
        assert p.get_tuning()["block_threads"] == block
        box, splits = np.array([[-2.0, 2.0]] * 2), np.array([70, 60], np.int32)
        F = p.enclose(box, splits, first=33, count=4001)[0]
    with ivb.Problem(tape(), specialize=0, autotune=0) as p:
        assert np.array_equal(F.view(np.uint8), p.enclose(box, splits, first=33, count=4001)[0].view(np.uint8))
