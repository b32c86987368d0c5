"""Pairs whose ids keep to their neighbourhood: a bucket's columns cover little of the id
range (graphs side by side, bands), or are one single column, or lie at both ends of the
range; and runs of equal pairs over many tiles.  Against the oracle's supergraph."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

MIN = 1 << 20  # edges from which the bucket sort runs


def _check(e, n):
    e = np.ascontiguousarray(e, np.int32)
    lab, dh = np.arange(n, dtype=np.int32), np.ones(n, np.uint32)
    sg, sg0 = (f(e, n, lab, dh, 1, 64, 5) for f in (G.supergraph, oracle.supergraph))
    assert sg["status"] == 0 and sg["K"] == sg0["K"] and sg["Es"] == sg0["Es"]
    for k in ("src", "dst", "w", "csr_off", "csr_adj", "csr_w"):
        assert np.array_equal(np.asarray(sg[k]).astype(np.int64), np.asarray(sg0[k]).astype(np.int64)), k


@pytest.mark.parametrize("n", [200, 5000, 40_000, 600_001])
@pytest.mark.parametrize("kind", ["blocks", "band", "ends", "column"])
def test_columns_in_a_small_range(n, kind):
    rng = np.random.default_rng(n)
    u = rng.integers(0, n, MIN + 5)
    if kind == "blocks":  # about 30 ids a graph
        v = u // 30 * 30 + rng.integers(0, 30, u.shape[0])
    elif kind == "band":
        v = u + rng.integers(-3, 4, u.shape[0])
    elif kind == "ends":
        v = np.where(rng.random(u.shape[0]) < 0.5, rng.integers(0, 3, u.shape[0]), n - 1 - rng.integers(0, 3, u.shape[0]))
    else:
        v = np.full(u.shape[0], n // 3)
    _check(np.stack([u, np.clip(v, 0, n - 1)], 1), n)


def test_runs_over_many_tiles():
    # two pairs that take 700,000 keys each beside a few others: tiles without a new pair
    rng = np.random.default_rng(2)
    e = np.concatenate([np.tile([[0, 1]], (700_000, 1)), np.tile([[2, 1]], (MIN - 700_000, 1)),
                        rng.integers(0, 5, (1000, 2))])
    _check(e[rng.permutation(e.shape[0])], 5)
    _check(np.tile([[3, 4]], (MIN + 1, 1)), 5)


def test_graphs_side_by_side_are_no_slower():
    # rows of about a hundred columns among a thousand ids took three times as long as over all ids
    n, m = 40_000, 3_000_000
    g = torch.Generator(device="cuda").manual_seed(1)
    u = torch.randint(n, (m,), generator=g, device="cuda")
    t = []
    for v in (torch.randint(n, (m,), generator=g, device="cuda"),
              u // 400 * 400 + torch.randint(400, (m,), generator=g, device="cuda")):
        e = torch.stack([u, v], 1).to(torch.int32).contiguous()
        out = [torch.zeros(k, dtype=torch.int32, device="cuda") for k in (n + 1, 2 * m, 2 * m, n)]
        nnz, ws = torch.zeros(1, dtype=torch.int64, device="cuda"), G.B.alloc_ws(G.B.bgv_graph_csr_ws_size(m, n))
        best = np.inf
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            G.B.bgv_graph_csr(e, m, n, *out, nnz, ws)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        t.append(best)
    assert t[1] < 1.4 * t[0], t
