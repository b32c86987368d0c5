"""The community rounds' bit map where a bit stands for up to 64 ids (from 16.8 M nodes),
where it is dropped (nearly every edge passes, from the first round or a later one), and
below the edges that use one, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import gpu_pipeline as G  # noqa: E402

MIN = 1 << 17  # edges from which a map is used


def _check(e, n, dh, passes, threshold, growth=2, tie=0):
    e = np.ascontiguousarray(e, np.int32)
    lab, deg, st = G.communities(e, n, dh, passes, threshold, growth, tie)
    lab0, deg0 = oracle.communities(e, n, dh, passes, threshold, growth, tie)
    assert st == 0 and np.array_equal(lab, lab0) and np.array_equal(deg, deg0)


# shifts 0, 1, 4, 5, 6: around 524,288 nodes a bit, and 32 or more a row
@pytest.mark.parametrize("n", [524_288, 524_289, 5_000_001, 8_388_609, 16_777_300])
@pytest.mark.parametrize("low", [0.0, 0.02, 0.5])
def test_ids_per_bit(n, low):
    rng = np.random.default_rng(n)
    e = rng.integers(0, n, (MIN + 3, 2))
    e[:MIN // 2] = (e[:MIN // 2] // 997) % 1009 + n - 1009  # many edges among few ids, the last among them
    dh = np.where(rng.random(n) < low, rng.integers(1, 9, n), rng.integers(100, 200, n)).astype(np.uint32)
    dh[n - 1009:] = rng.integers(1, 12, 1009)
    _check(e, n, dh, 4, 2, tie=1)


@pytest.mark.parametrize("m", [MIN - 1, MIN, MIN + 1])
@pytest.mark.parametrize("threshold,growth", [(1, 1), (3, 2), (9, 2), (1000, 2)])
def test_the_map_is_dropped(m, threshold, growth):
    # uniform degrees about 9: shares of 0 to 1, reached at once, after some rounds or never
    n = 2 * MIN // 9
    rng = np.random.default_rng(m)
    e = rng.integers(0, n, (m, 2))
    dh = np.bincount(e.reshape(-1), minlength=n).astype(np.uint32)
    _check(e, n, dh, 6, threshold, growth)
