"""The bucket sort of the supergraph's pairs (from 1,048,576 edges up) against
the oracle's supergraph, on the shapes that take its different ways: few
supernodes (bins of equal keys), rows spread out, hubs and repeated pairs that
fill whole bins, and keys too lopsided for it."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B
MIN = 1 << 20  # edges from which the bucket sort runs


def _check(e, n, lab, pad=True):
    e = np.ascontiguousarray(e, np.int32)
    if pad and e.shape[0] < MIN:  # loops have no pairs
        e = np.concatenate([e, np.zeros((MIN + 1 - e.shape[0], 2), np.int32)])
    dh = np.bincount(e.reshape(-1), minlength=n).astype(np.uint32)
    sg, sg0 = G.supergraph(e, n, lab, dh, 2, 512, 5), oracle.supergraph(e, n, np.asarray(lab, np.int32), dh, 2, 512, 5)
    assert sg["status"] == 0
    assert sg["K"] == sg0["K"] and sg["Es"] == sg0["Es"]
    for k in ("node_map", "src", "dst", "w", "mass", "vol", "count", "comm_label", "csr_off", "csr_adj", "csr_w"):
        assert np.array_equal(np.asarray(sg[k]).astype(np.int64), np.asarray(sg0[k]).astype(np.int64)), k


def _labels(rng, n, K):
    """K labels, each at least once."""
    lab = rng.choice(rng.permutation(n)[:K], n)
    lab[rng.permutation(n)[:K]] = np.unique(lab)[:1] if K == 1 else rng.permutation(n)[:K]
    return lab.astype(np.int32)


# around the least edge count; one supernode (no pairs), bins that are single keys (K <= 181), parts of rows
# (182 .. 32,768), whole rows; odd edge counts
@pytest.mark.parametrize("m", [MIN - 1, MIN, MIN + 1, 400_003, 1_400_003])
@pytest.mark.parametrize("K", [1, 2, 10, 181, 182, 300, 5000, 40_000])
def test_random_labels(m, K):
    n = 100_003
    rng = np.random.default_rng(K + m)
    e = rng.integers(0, n, (m, 2))
    lab = np.arange(n) if K == 1 and m == MIN else (np.zeros(n) if K == 1 else _labels(rng, n, K))
    _check(e, n, lab.astype(np.int32), pad=m != MIN - 1)


@pytest.mark.parametrize("n", [20_000, 1 << 17, 3_000_001])
@pytest.mark.parametrize("skew", [1.0, 6.0])
def test_identity_labels(n, skew):
    # every node its own supernode; skew 6: hubs whose rows fill whole bins and are split, some past 32 per bin
    rng = np.random.default_rng(n)
    m = 700_001
    e = np.minimum((rng.random((m, 2)) ** skew * n).astype(np.int64), n - 1)
    _check(e, n, np.arange(n, dtype=np.int32))


@pytest.mark.parametrize("n,hub", [(300_000, 0), (300_000, 299_999), (3_000_001, 1_234_567)])
def test_star(n, hub):
    # one row longer than a block sorts, split by its columns
    rng = np.random.default_rng(hub)
    leaves = rng.permutation(n)[:250_000]
    e = np.stack([np.full(leaves.shape[0], hub), leaves], 1)
    _check(e, n, np.arange(n, dtype=np.int32))


@pytest.mark.parametrize("copies", [30, 700, 5000, 30_000, 400_000])
def test_repeated_pairs(copies):
    # a few pairs many times among pairs that occur once: bins ranked, sorted by a warp, by a block, counted out
    n = 200_000
    rng = np.random.default_rng(copies)
    heavy = rng.integers(0, n, (max(1, min(60, 600_000 // copies)), 2))
    heavy = np.concatenate([heavy, heavy[:1] + 1])  # a neighbouring key too
    e = np.concatenate([np.repeat(np.minimum(heavy, n - 1), copies, axis=0), rng.integers(0, n, (200_000, 2))])
    _check(e[rng.permutation(e.shape[0])], n, np.arange(n, dtype=np.int32))


@pytest.mark.parametrize("n", [100_000, 9_000_000])
def test_one_pair_takes_nearly_all(n):
    # 2.4 M keys in one bin: the LSD sort takes over
    rng = np.random.default_rng(n)
    e = np.concatenate([np.tile([[0, 1]], (1_200_000, 1)), rng.integers(0, n, (150_000, 2))])
    _check(e[rng.permutation(e.shape[0])], n, np.arange(n, dtype=np.int32))


def test_dense_rows_of_a_large_id_space():
    # 24-bit ids: a bucket left over after both splits is counted in several slices
    n = 9_000_000
    rng = np.random.default_rng(5)
    e = np.stack([np.full(200_000, 4_000_000), 5_000_000 + rng.integers(0, 40_000, 200_000)], 1)
    _check(np.concatenate([e, rng.integers(0, n, (50_000, 2))]), n, np.arange(n, dtype=np.int32))


@pytest.mark.parametrize("identity", [True, False])
def test_bad_endpoints_are_reported(identity):
    n = 1000
    rng = np.random.default_rng(1)
    e = rng.integers(0, n, (MIN, 2)).astype(np.int32)
    e[77] = [5, n + 3]
    lab = np.arange(n) if identity else rng.integers(0, n, n)
    sg = G.supergraph(e, n, lab.astype(np.int32), np.ones(n, np.uint32), 1, 64, 1, optional=False)
    assert sg["status"] == B.BGV_DEV_BADEDGE
