"""Later steps of a run whose keys have moved as a whole since the step before (a tight
start that expands, a few far bodies that stretch the frame): many bodies lie between
two of the previous order's splitters, and the step counts again between samples of
its own keys.  Equal to the radix sort's steps bit for bit."""
import numpy as np
import pytest

import graphgen
from oracle import FA2Params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B


def _start(K, kind, rng):
    pos = rng.random((K, 2))
    if kind == "unit":
        return pos
    if kind == "tight":
        return rng.normal(size=(K, 2)) * 1e-2
    if kind == "far":  # ten bodies far off, drawn in step by step
        pos *= 100
        pos[:10] *= 50
        return pos
    pos[K // 2:] = pos[0]  # half of the bodies in one place: equal keys, told apart by id
    return pos * 1e-3


def _run(args, steps, order, replay):
    prev = B.bgv_set_fa2_order(order)
    try:
        dv, st = G.Fa2Device(*args), torch.cuda.Stream()
        dv.run(steps, replay, stream=st)
        torch.cuda.synchronize()
        return dv.state(), dv.stats()
    finally:
        B.bgv_set_fa2_order(prev)


# two buckets, a few, many; around the sorts' lines
@pytest.mark.parametrize("K", [2100, 9000, 40_003, 70_001, 300_007])
@pytest.mark.parametrize("kind", ["unit", "tight", "far", "half"])
def test_steps_agree(K, kind):
    if kind == "half" and K > 9000:
        pytest.skip("thousands of coincident bodies per leaf: slow")
    rng = np.random.default_rng(K)
    off, adj, w = G.csr_from_edges(graphgen.random_graph(K, 3 * K, seed=5), K)
    args = (_start(K, kind, rng).astype(np.float32), rng.integers(1, 9, K).astype(np.uint32), off, adj, w, FA2Params())
    want, sw = _run(args, 7, 0, False)
    for replay in (False, True):
        got, sg = _run(args, 7, 1, replay)
        assert sg.status == 0 and (sg.interactions, sg.tree_nodes) == (sw.interactions, sw.tree_nodes)
        for x, y in zip(got, want):
            assert np.array_equal(x, y)


def test_moved_keys_cost_about_a_sort():
    # a step of moved keys used to have one block merge most of the bodies: 30 times a usual step
    K = 400_000
    rng = np.random.default_rng(1)
    off, adj, w = G.csr_from_edges(graphgen.random_graph(K, 2 * K, seed=2), K)
    ms = {}
    for kind in ("usual", "tight"):
        pos = rng.normal(size=(K, 2)) * (1e-2 if kind == "tight" else 1e3)
        dv = G.Fa2Device(pos.astype(np.float32), np.ones(K, np.uint32), off, adj, w, FA2Params())
        best = np.inf
        for _ in range(4):
            dv.pos.copy_(G.dev(pos.astype(np.float32)))
            dv.Fprev.zero_()
            dv.speed.fill_(1.0)
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            dv.run(3, False)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ms[kind] = best
    assert ms["tight"] < 4 * ms["usual"], ms
