"""Graphs of up to 2,048 bodies, whose runs stay in the shared memory of one
cluster of blocks, against the general path (bgv_fa2_run_timed launches its
kernels step by step whatever the size): equal bits."""
import numpy as np
import pytest

import graphgen
import oracle
from oracle import FA2Params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B


def _general(dv, steps):
    B.bgv_fa2_run_timed(dv.K, dv.nnz, dv.off, dv.adj, dv.w, dv.mass, dv.params, steps, dv.pos, dv.F, dv.Fprev,
                        dv.speed, dv.ws)


def _same(a, b):
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y, equal_nan=True)
    s, t = a.stats(), b.stats()
    assert s.status == 0 and t.status == 0
    for f in ("S", "T", "interactions", "tree_nodes", "interactions_total", "steps_total"):
        assert getattr(s, f) == getattr(t, f), f


def _graph(K, degree, seed, weight=5):
    rng = np.random.default_rng(seed)
    e = graphgen.random_graph(K, K * degree // 2, seed=seed) if K > 1 else np.zeros((0, 2), np.int32)
    off, adj, w = G.csr_from_edges(e, K)
    w = rng.integers(1, weight, w.shape[0]).astype(np.uint32)
    return rng.integers(1, 50, K).astype(np.uint32), off, adj, w


# one body, around the cluster sizes (128, 256, 512 bodies) and the largest; no edges, rows of one lane and of a warp
@pytest.mark.parametrize("K", [1, 2, 3, 31, 128, 129, 256, 257, 512, 513, 1000, 1764, 2047, 2048])
@pytest.mark.parametrize("degree", [0, 6, 60])
def test_runs_equal_the_general_path(K, degree):
    args = (oracle.fa2_init(K, 3), *_graph(K, degree, K + degree), FA2Params())
    small, general = G.Fa2Device(*args), G.Fa2Device(*args)
    small.run(7, True)
    _general(general, 7)
    _same(small, general)
    small.step()
    _general(general, 1)
    _same(small, general)


@pytest.mark.parametrize("prm", [dict(theta=0.0), dict(theta=0.7, leaf_cap=6), dict(max_depth=3), dict(strong_gravity=1),
                                 dict(kr=80.0, leaf_cap=64, max_depth=9)])
def test_parameters(prm):
    args = (oracle.fa2_init(700, 5), *_graph(700, 8, 1), FA2Params(**prm))
    small, general = G.Fa2Device(*args), G.Fa2Device(*args)
    small.run(5, False)
    _general(general, 5)
    _same(small, general)


@pytest.mark.parametrize("layout", ["coincident", "clump", "line", "nan"])
def test_layouts(layout):
    # many keys in one bin of the sort, equal keys, deep chains, a position that is not a number
    K = 1500
    rng = np.random.default_rng(2)
    pos = rng.random((K, 2)) * 100
    if layout == "coincident":
        pos[:900] = pos[rng.integers(0, 5, 900)]
    elif layout == "clump":
        pos[5:] = pos[5] + rng.normal(size=(K - 5, 2)) * 1e-3
    elif layout == "line":
        pos[:, 0] = 2.0 ** -rng.uniform(0, 22, K)
        pos[:, 1] = pos[:, 0] / 2
    else:
        pos[77] = np.nan
    args = (pos.astype(np.float32), *_graph(K, 10, 4), FA2Params())
    steps = 1 if layout == "nan" else 4
    small, general = G.Fa2Device(*args), G.Fa2Device(*args)
    small.run(steps, False)
    _general(general, steps)
    if layout == "nan":
        assert np.array_equal(small.state()[1], general.state()[1], equal_nan=True)
    else:
        _same(small, general)


def test_rows_that_do_not_fit_and_rows_of_a_block():
    # more entries than a block keeps, a weight too wide for its cache, a row longer than a warp takes
    K = 300
    rng = np.random.default_rng(9)
    lengths = rng.integers(0, 90, K)
    lengths[7], lengths[200] = 5000, 9000
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    adj = rng.integers(-1, K + 1, off[-1]).astype(np.int32)  # some outside [0, K): they add nothing
    for wide in (5, 1 << 30):
        w = rng.integers(1, wide, off[-1]).astype(np.uint32)
        args = (oracle.fa2_init(K, 3), np.ones(K, np.uint32), off, adj, w, FA2Params())
        small, general = G.Fa2Device(*args), G.Fa2Device(*args)
        small.run(3, False)
        _general(general, 3)
        _same(small, general)


def test_more_steps_than_one_launch():
    args = (oracle.fa2_init(150, 3), *_graph(150, 6, 1), FA2Params())
    one, two = G.Fa2Device(*args), G.Fa2Device(*args)
    one.run(600, True)
    two.run(255, True)
    two.run(345, False)
    _same(one, two)


@pytest.mark.parametrize("sizes", [[1, 1], [5, 300, 1, 128, 2048], [200] * 30])
def test_batches_equal_each_graph_alone(sizes):
    parts = [(oracle.fa2_init(k, i + 1), *_graph(k, 6, i)) for i, k in enumerate(sizes)]
    koff = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    nnz = np.concatenate([[0], np.cumsum([p[2][-1] for p in parts])])
    off = np.concatenate([[0]] + [p[2][1:] + nnz[i] for i, p in enumerate(parts)]).astype(np.int32)
    adj = np.concatenate([p[3] + koff[i] for i, p in enumerate(parts)]).astype(np.int32)
    P = G.dev(np.concatenate([p[0] for p in parts]).astype(np.float32))
    F, Fp = torch.zeros_like(P), torch.zeros_like(P)
    sp = torch.ones(len(sizes), dtype=torch.float64, device="cuda")
    ws = B.alloc_ws(B.bgv_fa2_ws_size_batched(len(sizes), int(koff[-1]), int(nnz[-1])))
    B.bgv_fa2_run_batched(len(sizes), koff, int(nnz[-1]), G.dev(off), G.dev(adj),
                          G.dev(np.concatenate([p[4] for p in parts])), G.dev(np.concatenate([p[1] for p in parts])),
                          G.fa2_params(FA2Params()), 5, True, P, F, Fp, sp, ws)
    inter = 0
    for g in range(len(sizes)):
        one = G.Fa2Device(*parts[g], FA2Params())
        _general(one, 5)
        pos, f, _, speed = one.state()
        inter += one.stats().interactions
        rows = slice(koff[g], koff[g + 1])
        assert np.array_equal(G.host(P)[rows], pos.astype(np.float32))
        assert np.array_equal(G.host(F)[rows], f.astype(np.float32)) and float(sp[g]) == speed
    assert B.bgv_fa2_read_stats(ws).interactions == inter and B.bgv_fa2_read_stats(ws).steps_total == 5
