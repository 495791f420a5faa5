"""ES_pool's enumeration at the sizes where its sweeps change shape, against the
fp64 oracle: one batch or several of the smaller side's subsets, 1 to 9 and
more exchanged keys (the unrolled and the general member loops), odd and full
pools, rows whose best subsets leave out the sink (swept again around them),
rows of equal values (every subset scored), non-finite rows and pools whose
products leave the range fp32 squares hold."""
import itertools
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


def test_rows_without_an_answer(fw):  # noqa: F811
    # a NaN or infinite logit, or value, leaves no es to compare: the row is reported
    # and nothing is enumerated (a pool of 1.9e9 subsets a row)
    L, V = _rows(3, 8, 100, 32, 2.0, 1.0)
    L[0, 50], L[1, 7], L[2, 8] = np.nan, np.inf, -np.inf
    V[3, 60, 5], V[4, 0, 31], V[5, 2, 0] = np.nan, np.inf, -np.inf
    _, out = run_pool(fw, rows_batch(L, V, np.tile(np.array([15, 32], np.int32), (8, 1))), [19, 2])
    assert list(np_(out["row_status"])) == [fw.FW_ERR_NONFINITE] * 6 + [0, 0]
    for key in ("best_gap", "topk_gap"):
        assert np.isnan(np_(out[key])[:6]).all() and np.isfinite(np_(out[key])[6:]).all()
    assert (np_(out["best_idx"])[:6] == -1).all() and not np_(out["n_cand"])[:6].any()


@pytest.mark.parametrize("sink,scale", [(36.0, 1.0), (40.0, 1.0), (5.0, 2.0 ** -55), (5.0, 2.0 ** 55)])
def test_pools_far_from_unit_scale(fw, sink, scale):  # noqa: F811
    # masses of 1e-17 beside a sink that the dense output equals, and small and large
    # values: the sets of fp64, and few of the subsets scored
    L, V = _rows(17, 6, 60, 64, sink, 1.0)
    V = (np.round(V * 8) / 8).astype(np.float32) * np.float32(scale)
    b = rows_batch(L, V, np.full((6, 1), 4))
    rows, out = run_pool(fw, b, [24])
    top = fw.dense_and_topk_gap(rows, torch.full((6, 1), 4, dtype=torch.int32).cuda())
    o, gap, idx = (np_(x).astype(np.float64) for x in (top["o"], out["best_gap"], out["best_idx"]))
    assert not np_(out["row_status"]).any()
    for r in range(6):
        p = np.exp(L[r].astype(np.float64) - L[r].max())
        u = p[:, None] / p.sum() * (V[r].astype(np.float64) - o[r])  # (the gap call's output, as the pool takes it)
        e = np.linalg.norm(u, axis=1)
        kept = np.lexsort((np.arange(60), -L[r].astype(np.float64)))[:4]
        e[kept] = np.inf
        pool = np.sort(np.argsort(-e, kind="stable")[:28])
        sets = np.array(list(itertools.combinations(pool, 4)))
        es = np.linalg.norm(u[sets].sum(1), axis=1) / (p[sets] / p.sum()).sum(1)
        best = es.argmin()
        assert abs(gap[r, 0] - es[best]) <= 1e-5 * es[best]
        if np.partition(es, 1)[1] > es[best] * (1 + 1e-5):
            np.testing.assert_array_equal(idx[r, 0, :4], sets[best])
    assert np_(out["n_cand"]).max() <= 600  # (of 20,475)
