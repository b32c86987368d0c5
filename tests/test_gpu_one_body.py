"""A single body has no tree: its counters are its own, whatever the workspace held."""
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


@pytest.mark.parametrize("call", ["forces", "run_timed", "step", "run"])
@pytest.mark.parametrize("order", [0, 1])
def test_counters_after_a_larger_graph(call, order):
    K = 900
    off, adj, w = G.csr_from_edges(graphgen.random_graph(K, 3 * K, seed=1), K)
    many = G.Fa2Device(oracle.fa2_init(K, 1), np.ones(K, np.uint32), off, adj, w, FA2Params())
    one = G.Fa2Device(np.array([[3.0, 4.0]], np.float32), np.ones(1, np.uint32), np.zeros(2, np.int32),
                      np.zeros(0, np.int32), np.zeros(0, np.uint32), FA2Params())
    prev = B.bgv_set_fa2_order(order)
    try:
        for dv in (many, one):
            args = (dv.K, dv.nnz, dv.off, dv.adj, dv.w, dv.mass, dv.params)
            if call == "forces":
                out = [torch.empty_like(dv.pos) for _ in range(3)]
                B.bgv_fa2_forces(*args, dv.pos, *out, many.ws)
            elif call == "run_timed":
                B.bgv_fa2_run_timed(*args, 2, dv.pos, dv.F, dv.Fprev, dv.speed, many.ws)
            elif call == "step":
                B.bgv_fa2_step(*args, dv.pos, dv.F, dv.Fprev, dv.speed, many.ws)
            else:
                B.bgv_fa2_run(*args, 3, False, dv.pos, dv.F, dv.Fprev, dv.speed, many.ws)
            st = B.bgv_fa2_read_stats(many.ws)
            assert st.status == 0
            if dv is many:
                assert st.interactions > 0 and st.tree_nodes > 0
            else:
                assert st.interactions == 0 and st.tree_nodes == 0
    finally:
        B.bgv_set_fa2_order(prev)
