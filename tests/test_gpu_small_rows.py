"""Rows of graphs of up to 2,048 bodies that lie unevenly: hubs side by side (one warp's
nodes), more entries than a block keeps, weights too wide to keep, rows of more than
4,096 entries, and the most entries a small graph may have (131,072).  Equal to the
general path bit for bit, and no slower than a larger graph."""
import numpy as np
import pytest

import oracle
from oracle import FA2Params

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B


def _hubs(K, hubs, entries, rng):
    """Symmetric CSR: `hubs` neighbouring nodes with most of the entries."""
    u, v = rng.integers(0, hubs, entries // 2), rng.integers(0, K, entries // 2)
    return G.csr_from_edges(np.unique(np.sort(np.stack([u, v], 1), 1), axis=0), K)


def _same(args, steps):
    small, general = G.Fa2Device(*args), G.Fa2Device(*args)
    small.run(steps, False)
    B.bgv_fa2_run_timed(general.K, general.nnz, general.off, general.adj, general.w, general.mass, general.params, steps,
                        general.pos, general.F, general.Fprev, general.speed, general.ws)
    assert small.stats().status == 0 and general.stats().status == 0
    for x, y in zip(small.state(), general.state()):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("K,hubs,entries", [(128, 1, 250), (129, 32, 8000), (300, 40, 20_000), (1000, 17, 30_000),
                                            (1500, 187, 100_000), (2048, 256, 120_000)])
@pytest.mark.parametrize("weight", [5, 1 << 22])
def test_hubs_side_by_side(K, hubs, entries, weight):
    rng = np.random.default_rng(K)
    off, adj, w = _hubs(K, hubs, entries, rng)
    w = rng.integers(1, weight, w.shape[0]).astype(np.uint32)
    _same((oracle.fa2_init(K, 3), rng.integers(1, 9, K).astype(np.uint32), off, adj, w, FA2Params()), 4)


@pytest.mark.parametrize("length", [32, 33, 4096, 4097, 9000, 100_001])
def test_one_long_row(length):
    K = 500
    rng = np.random.default_rng(length)
    lens = rng.integers(0, 40, K)
    lens[77] = length  # neighbours repeat
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    adj = rng.integers(0, K, off[-1]).astype(np.int32)
    _same((oracle.fa2_init(K, 1), np.ones(K, np.uint32), off, adj, np.ones(off[-1], np.uint32), FA2Params()), 3)


@pytest.mark.parametrize("nnz", [(1 << 17) - 1, 1 << 17, (1 << 17) + 1])
def test_the_most_entries(nnz):
    K = 2048
    rng = np.random.default_rng(nnz)
    off = np.sort(rng.integers(0, nnz + 1, K + 1)).astype(np.int32)
    off[0], off[-1] = 0, nnz
    adj = rng.integers(0, K, nnz).astype(np.int32)
    _same((oracle.fa2_init(K, 1), np.ones(K, np.uint32), off, adj, rng.integers(1, 4, nnz).astype(np.uint32), FA2Params()), 3)


@pytest.mark.parametrize("K,entries", [(400, 36_000), (1500, 120_000), (1500, 240_000)])
def test_no_slower_than_a_larger_graph(K, entries):
    # 100 steps of hubs in an eighth of the rows used to take three times those of 2,049 bodies
    ms = []
    for n in (K, 2049):
        off, adj, w = _hubs(n, K // 8, entries, np.random.default_rng(1))
        dv = G.Fa2Device(oracle.fa2_init(n, 3), np.ones(n, np.uint32), off, adj, w, FA2Params())
        times = []
        for _ in range(4):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            dv.run(100, False)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        ms.append(min(times[1:]))
    assert ms[0] < 1.6 * ms[1], ms
