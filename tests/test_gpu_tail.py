"""The step's tail: nodes shared out in warp-sized chunks, the batched form's
per-graph sums, and the frame that a run's later steps take from the tail of
the step before.  A run (frames from the tail) must equal single steps (a frame
kernel each) bit for bit, and a batch each graph's own run."""
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


def _case(K, seed):
    e = graphgen.random_graph(K, 2 * K, seed=seed) if K > 2 else np.zeros((0, 2), np.int32)
    off, adj, w = G.csr_from_edges(e, K)
    mass = (np.diff(off) + 1).astype(np.uint32)
    return oracle.fa2_init(K, seed), mass, off, adj, w


# one node, around a warp row (32), a lane's items (128), a block (1,024), and a grid of several blocks
@pytest.mark.parametrize("K", [1, 2, 31, 33, 127, 129, 1023, 1024, 1025, 33_333])
def test_run_equals_single_steps(K):
    pos, mass, off, adj, w = _case(K, 7)
    run, steps = (G.Fa2Device(pos, mass, off, adj, w, FA2Params()) for _ in range(2))
    run.run(4, False)
    for _ in range(4):
        steps.step()
    a, b = run.state(), steps.state()
    assert run.stats().status == 0
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    assert run.stats().S == steps.stats().S and run.stats().T == steps.stats().T


# graphs of one body, graphs that end inside, on and past a warp's share, many tiny graphs, one large among them
@pytest.mark.parametrize("sizes", [[1, 1], [31, 1, 32, 33, 1, 128], [1000, 24, 1024, 1, 5000], [3] * 700 + [20_000] + [40] * 90])
def test_batch_equals_each_graph_alone(sizes):
    parts = [_case(k, 11 + i) for i, k in enumerate(sizes)]
    koff = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    K = int(koff[-1])
    off = np.concatenate([[0]] + [p[2][1:] + sum(q[2][-1] for q in parts[:i]) for i, p in enumerate(parts)])
    adj = np.concatenate([p[3] + koff[i] for i, p in enumerate(parts)]).astype(np.int32)
    w = np.concatenate([p[4] for p in parts]).astype(np.uint32)
    nnz, Gn = int(off[-1]), len(sizes)
    prm = G.fa2_params(FA2Params())
    O, A, W, M = G.dev(off.astype(np.int32)), G.dev(adj), G.dev(w), G.dev(np.concatenate([p[1] for p in parts]))
    P = G.dev(np.concatenate([p[0] for p in parts]).astype(np.float32))
    F, Fp = torch.zeros_like(P), torch.zeros_like(P)
    sp = torch.ones(Gn, dtype=torch.float64, device="cuda")
    ws = B.alloc_ws(B.bgv_fa2_ws_size_batched(Gn, K, nnz))
    B.bgv_fa2_run_batched(Gn, koff, nnz, O, A, W, M, prm, 3, False, P, F, Fp, sp, ws)
    assert B.bgv_fa2_read_stats(ws).status == 0
    P, F, sp = G.host(P), G.host(F), G.host(sp)
    for g in sorted({0, 1, Gn // 2, Gn - 2, Gn - 1} | {int(np.argmax(sizes))}):
        one = G.Fa2Device(*parts[g], FA2Params())
        one.run(3, False)
        pos, f, _, speed = one.state()
        rows = slice(koff[g], koff[g + 1])
        assert np.array_equal(P[rows], pos.astype(np.float32)) and np.array_equal(F[rows], f.astype(np.float32))
        assert sp[g] == speed
