"""The small-row kernels that stage 64 dimensions at a time and take the Gram
matrix in 4 x 4 tiles, at the row counts where the last tile is partial, for
every chunk count, against the fp64 oracle: swaps of several budgets with the
whole and a restricted pool, batches of more than 32 re-scored pairs, and the
best subset."""
import numpy as np
import pytest

from tests.test_gpu_small import check_best, check_swap, fw, rows_batch  # noqa: F401  (fw is a fixture)

pytestmark = pytest.mark.gpu


def _rows(n, d, rows, seed, v_dtype="f32", k=None):
    rng = np.random.default_rng(seed)
    L = (rng.gumbel(size=(rows, n)) * rng.uniform(0.3, 3, size=(rows, 1))).astype(np.float32)
    L[:, 0] += 5
    V = rng.normal(size=(rows, n, d)).astype(np.float32)
    if v_dtype == "bf16":
        V = (V.view(np.uint32) & 0xFFFF0000).view(np.float32)
    return rows_batch(L, V, np.tile(np.array(k, np.int32), (rows, 1)), v_dtype)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 8, 27, 28, 29, 31, 32])
@pytest.mark.parametrize("d", [32, 64, 128, 256])
def test_swap_tiles(fw, n, d):  # noqa: F811
    ks = [max(1, n // 4), max(1, n // 2), n, max(1, n - 1)]
    b = _rows(n, d, 21, 100 * n + d, "bf16" if n % 2 else "f32", ks)
    check_swap(fw, b, E=n, max_swaps=64)
    check_swap(fw, b, E=max(0, n // 5), max_swaps=64)


@pytest.mark.parametrize("n,k,d", [(3, 2, 32), (7, 3, 256), (8, 4, 32), (11, 5, 128), (15, 4, 64), (23, 5, 256),
                                   (24, 3, 32), (27, 2, 128), (28, 2, 64), (31, 2, 128), (32, 2, 256)])
def test_best_tiles(fw, n, k, d):  # noqa: F811
    check_best(fw, _rows(n, d, 9, n * d + k, "bf16" if k % 2 else "f32", [k]))


@pytest.mark.parametrize("copies,m,n,k", [(1, 1, 14, 4), (3, 1, 14, 4), (374, 13, 14, 4), (375, 13, 14, 4), (749, 13, 14, 4),
                                          (375, 13, 29, 2), (375, 13, 30, 2), (375, 13, 32, 3)])
def test_best_lanes_per_row(fw, copies, m, n, k):  # noqa: F811
    # 8 lanes walk a row up to 4,864 rows (152 SMs), 4 up to 9,728, or 2 where the walk
    # tables are large, and 2 beyond: the same few rows, repeated, give the same answers, and cost the same
    # search, as in a batch of their own
    import torch

    b = _rows(n, 32, m, 1000 * n + m, k=[k])
    rep = np.tile(np.arange(m), copies)
    big = rows_batch(np.asarray(b.logits).reshape(m, n)[rep], np.asarray(b.v).reshape(m, n, 32)[rep], np.asarray(b.k)[rep])
    check_best(fw, b)
    rows = [fw.rows_from_batch(x) for x in (b, big)]
    few, many = (fw.best_subset(r, torch.from_numpy(np.ascontiguousarray(x.k[:, 0])).cuda()) for r, x in zip(rows, (b, big)))
    for key in ("best_rank", "best_gap", "best_idx", "topk_gap"):
        np.testing.assert_array_equal(many[key].cpu().numpy(), few[key].cpu().numpy()[rep])
    one, all_ = (fw.best_subset_stats(r, o) for r, o in zip(rows, (few, many)))
    assert all_ == {key: copies * v for key, v in one.items()} and one["inner_leaves"] > 0


def test_swap_rescored_in_batches(fw):  # noqa: F811
    # equal logits and nearly equal values: the screen cannot tell the 240 pairs of a
    # row apart, so they are re-scored 32 at a time; the decision is the oracle's
    # wherever its margin is not a tie
    rng = np.random.default_rng(5)
    rows, n, d = 17, 32, 64
    L = np.zeros((rows, n), np.float32)
    L[:, 0] = 3
    V = (1 + 1e-4 * rng.normal(size=(rows, n, d))).astype(np.float32)
    V[:, 0] = rng.normal(size=(rows, d))
    check_swap(fw, rows_batch(L, V, np.full((rows, 1), 12)), E=n, max_swaps=32)
