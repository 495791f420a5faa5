"""ES_pool's enumeration at the sizes where its sweeps change shape, against the
fp64 oracle: one batch or several of the smaller side's subsets, 1 to 9 and
more exchanged keys (the unrolled and the general member loops), odd and full
pools, rows whose best subsets leave out the sink (swept again around them)
and rows of equal values (every subset scored)."""
import math

import numpy as np
import pytest

from tests.parity import np_
from tests.test_gpu_pool import check_pool, fw, run_pool  # noqa: F401  (fw is a fixture)
from tests.test_gpu_small import rows_batch

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _rows(seed, rows, n, d, sink, tau):
    rng = np.random.default_rng(seed)
    L = (rng.normal(size=(rows, n)) * tau).astype(np.float32)
    L[:, 0] += sink
    return L, rng.normal(size=(rows, n, d)).astype(np.float32)


# (s, E): 10 of 20 and 9 of 18 take several batches and the general loops; 1 of
# 64 and 60 extras are the widest sides; 7 + 6 and 5 + 8 are odd pools
@pytest.mark.parametrize("s,E", [(10, 10), (9, 9), (1, 63), (3, 60), (8, 8), (7, 6), (5, 8), (2, 1), (31, 3)])
@pytest.mark.parametrize("d,v_dtype", [(64, "bf16"), (32, "f32")])
def test_sweep_shapes(fw, s, E, d, v_dtype):  # noqa: F811
    L, V = _rows(100 * s + E, 4, 150, d, 5.0, 1.5)
    check_pool(fw, rows_batch(L, V, np.full((4, 1), s), v_dtype=v_dtype), [E])


@pytest.mark.parametrize("tau", [0.2, 1.0, 4.0])
def test_sink_heavy_rows(fw, tau):  # noqa: F811
    # the sink holds most of the kept mass: good subsets leave it out
    L, V = _rows(int(10 * tau), 12, 700, 128, 7.0, tau)
    k = np.tile(np.array([4, 8, 16, 32], np.int32), (12, 1))
    check_pool(fw, rows_batch(L, V, k, v_dtype="bf16"), [24, 12, 6, 4])


def test_every_subset_ties(fw):  # noqa: F811
    # equal values: every one of the C(14, 6) subsets has es = |v - o|, more
    # hits than the list holds, so the lanes score them all
    rng = np.random.default_rng(5)
    L = rng.normal(size=(2, 40)).astype(np.float32)
    V = np.tile(rng.normal(size=(2, 1, 64)).astype(np.float32), (1, 40, 1))
    b = rows_batch(L, V, np.full((2, 1), 6))
    _, out = run_pool(fw, b, [8])
    assert np.all(np_(out["n_cand"]) == math.comb(14, 6))
    check_pool(fw, b, [8], out=out)


def test_sums_that_need_52_bits(fw):  # noqa: F811
    # equal masses, o = 0.  The best subsets are {4, 5, 6} with key 1 or with key 0: the
    # first column sums to 1 or to 1 + 2^-24, beside terms of 2^27 that cancel.  Sums
    # of fewer than 52 bits make it a tie, which key 0 (the smaller rank) would win
    V = np.zeros((1, 8, 32), np.float32)
    V[0, :, 0] = [2.0 ** -24, 0, -(2.0 ** -24), 0, 2.0 ** 27, 1, -(2.0 ** 27), -1]
    V[0, :, 1] = [0, 0, 0, 30, 100, -200, 100, -30]
    V[0, :, 2] = [0, 0, 50, -50, 0, 0, 0, 0]
    b = rows_batch(np.zeros((1, 8), np.float32), V, [[4]])
    rows, out = run_pool(fw, b, [3])
    top = fw.dense_and_topk_gap(rows, torch.tensor([[4]], dtype=torch.int32).cuda())
    assert not np_(top["o"]).any()
    np.testing.assert_array_equal(np_(out["best_idx"])[0, 0, :4], [1, 4, 5, 6])
    assert float(np_(out["best_gap"])[0, 0]) == 0.25
