"""Community rounds behind the bit map of nodes that pass the threshold: one
id per bit (from 131,072 edges up; without the map below), several ids per bit (more ids than the map has bits), rounds that
no node passes before rounds that some do, and bad endpoints when no node passes."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B

MAP_BITS = 208 * 1024 * 8


@pytest.mark.parametrize("n,m", [(1, 0), (31, 60), (33, 61), (128, 400), (1025, 4001), (40_000, 160_001), (33, 1 << 17), (1025, (1 << 17) + 1),
                                 (40_000, (1 << 17) - 1), (40_000, 300_001),
                                 (MAP_BITS, 800_000), (MAP_BITS + 1, 800_001), (4 * MAP_BITS + 5, 2_000_001)])
@pytest.mark.parametrize("threshold,tie", [(0, 1), (1, 0), (6, 1)])
def test_rounds_match_oracle(n, m, threshold, tie):
    rng = np.random.default_rng(n)
    # skewed endpoints, some loops and repeats: degrees from 0 to thousands
    e = np.minimum((rng.random((m, 2)) ** 1.5 * n).astype(np.int64), n - 1).astype(np.int32)
    deg = np.bincount(e.reshape(-1), minlength=n).astype(np.uint32)
    lab, d, st = G.communities(e, n, deg, 4, threshold, 2, tie)
    lab0, d0 = oracle.communities(e, n, deg, 4, threshold or (2 * m) // n, 2, tie)
    assert st == 0
    assert np.array_equal(lab, lab0) and np.array_equal(d, d0)


@pytest.mark.parametrize("copies", [1, 7])  # 7: enough edges for the map
def test_rounds_that_nothing_passes_come_before_rounds_that_move(copies):
    n, e, _ = graphgen.load("sbm16")
    deg = np.bincount(e.reshape(-1), minlength=n).astype(np.uint32) + 50
    e = np.tile(e, (copies, 1))
    lab, d, st = G.communities(e, n, deg, 8, 1, 2, 0)  # thresholds 1, 2, 4, ..., 128: degrees start at 50
    lab0, d0 = oracle.communities(e, n, deg, 8, 1, 2, 0)
    assert st == 0 and (lab0 != np.arange(n)).any()
    assert np.array_equal(lab, lab0) and np.array_equal(d, d0)


def test_bad_endpoints_are_reported_when_no_node_passes():
    e = np.array([[0, 1], [2, 3], [5, 107], [4, 6]], np.int32)
    _, _, st = G.communities(e, 100, np.full(100, 9, np.uint32), 2, 1)
    assert st == B.BGV_DEV_BADEDGE


def test_batched_rounds_with_several_ids_per_bit():
    sizes = [MAP_BITS // 2, 5, MAP_BITS // 2 + 77, 1000]
    parts = [graphgen.random_graph(n, n // 2 if n > 2000 else 2 * n, seed=3 + i) for i, n in enumerate(sizes)]
    node_off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    edge_off = np.concatenate([[0], np.cumsum([p.shape[0] for p in parts])]).astype(np.int64)
    p = B.bgv_layout_default_params()
    p.iterations, p.threshold, p.tie_mode = 0, 3, 1
    N = int(node_off[-1])
    E, _ = G.edges_dev(np.concatenate(parts))
    nm = G.empty(N, np.int32)
    xy, rad = torch.zeros((N, 2), device="cuda"), torch.zeros(N, device="cuda")
    ws = B.alloc_ws(B.bgv_layout_batched_ws_size(len(sizes), edge_off, node_off, p))
    B.bgv_layout_batched(E, len(sizes), edge_off, node_off, p, nm, xy, rad, ws)
    nm = G.host(nm)
    for i, n in enumerate(sizes):
        _, dh = oracle.sketch_degrees(parts[i], n, 4, 4096, 1)
        lab, _ = oracle.communities(parts[i], n, dh, 3, 3, 2, 1)
        _, ref = np.unique(lab, return_inverse=True)
        assert np.array_equal(nm[node_off[i]:node_off[i + 1]], ref)
