"""The TMA-fed P.V kernel at the stage counts where its producer sets and chunk
flushes end differently (64-key stages, two sets of producer warps, chunks of
8 stages), for the gap call and the group vote, ties at the thresholds
included, against the fp64 oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
from tests.test_gpu_long import compare, fw  # noqa: F401  (fw is a fixture)
from tests.test_gpu_small import rows_batch
from tests.test_gpu_vote import check_vote, group_budgets, run_vote

pytestmark = pytest.mark.gpu


def _batch(n, d, R, ks, ties, seed):
    rng = np.random.default_rng(seed)
    L = (rng.normal(size=(R, n)) * 1.5).astype(np.float32)
    L[:, 0] += 5
    if ties:
        L = (np.round(L * 8) / 8).astype(np.float32)  # every threshold has equal keys, some dropped
    V = rng.normal(size=(1, n, d)).astype(np.float32)
    return rows_batch(L, V, np.tile(np.asarray(ks, np.int32), (R, 1)), v_dtype="bf16", R=R)


# stages 1..11 and 16..19: both sets' last stages, with and without a chunk end near them
@pytest.mark.parametrize("stages", [1, 2, 3, 7, 8, 9, 10, 11, 16, 17, 18, 19])
@pytest.mark.parametrize("d", [64, 128])
def test_stage_counts(fw, stages, d):  # noqa: F811
    for n in (64 * stages, 64 * stages - 31):
        ks = [max(1, n // 2), max(1, n // 9), n][: 1 + stages % 3]  # not in order
        compare(fw, _batch(n, d, 34, ks, stages % 2 == 0, n + d))


@pytest.mark.parametrize("n", [64 * 3, 64 * 17 - 5])
def test_vote_stage_counts(fw, n):  # noqa: F811
    b = _batch(n, 128, 20, [n // 4, n // 16, n // 2], True, n)
    s = group_budgets(b)
    _, _, v = run_vote(fw, b, s)
    check_vote(oracle.HostRows(b), s, v)


@pytest.mark.parametrize("n", [64 * 2, 64 * 9 + 1, 64 * 21 - 31])
@pytest.mark.parametrize("d", [64, 128])
def test_value_blocks_off_whole_rows(fw, n, d):  # noqa: F811
    # v_off not a multiple of d: no stage's values can come by TMA, every one is
    # copied by threads (one of the groups stays on whole rows)
    R, G = 20, 3
    rng = np.random.default_rng(n + d)
    L = (rng.normal(size=(G * R, n)) * 1.5).astype(np.float32)
    V = rng.normal(size=(G, n, d)).astype(np.float32)
    b = rows_batch(L, V, np.tile(np.array([n // 3, n // 20 + 1], np.int32), (G * R, 1)), v_dtype="bf16", R=R)
    off = np.array([8, n * d + d - 8, 2 * n * d + 2 * d], np.int64)
    v = np.zeros(3 * n * d + 3 * d, b.v.dtype)
    for g in range(G):
        v[off[g]:off[g] + n * d] = b.v[g * n * d:(g + 1) * n * d]
    b = dataclasses.replace(b, v=v, v_off=off)
    compare(fw, b)
    s = group_budgets(b)
    _, _, o = run_vote(fw, b, s)
    check_vote(oracle.HostRows(b), s, o)
