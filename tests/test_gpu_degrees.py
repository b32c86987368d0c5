"""Degrees counted by node ranges (from 4,194,304 edges up, to 16,777,216 nodes)
against NumPy, around the ranges of 32,768 nodes and the smallest edge count."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

B = G.B


@pytest.mark.parametrize("m", [(1 << 22) - 1, 1 << 22, (1 << 22) + 1, 5_234_567])
@pytest.mark.parametrize("n,skew", [(1, 1.0), (32_767, 1.0), (32_768, 5.0), (32_769, 1.0), (400_001, 3.0),
                                    (16_777_216, 1.0), (16_777_217, 1.0)])
def test_sketch_over_node_ranges(n, m, skew):
    rng = np.random.default_rng(n + m)
    e = np.minimum((rng.random((m, 2)) ** skew * n).astype(np.int64), n - 1).astype(np.int32)
    S, d, st = G.sketch(e, n, 2, 4096, 3)
    S0, d0 = oracle.sketch_degrees(e, n, 2, 4096, 3)
    assert st == 0 and np.array_equal(S, S0) and np.array_equal(d, d0)


def test_one_node_takes_every_endpoint_and_bad_ones_are_reported():
    n, m = 100_000, 4_700_001
    e = np.full((m, 2), 65_536, np.int32)
    S, d, st = G.sketch(e, n, 1, 4096, 3)
    assert st == 0 and np.array_equal(S, oracle.sketch_degrees(e, n, 1, 4096, 3)[0])
    e[m - 1] = [n, -1]
    assert G.sketch(e, n, 1, 4096, 3)[2] == B.BGV_DEV_BADEDGE
