"""The long-row swap kernel where its bounds and branches change: extras that do
not fill a lane's eight slots, several blocks of 32 slots, rows whose sink
holds nearly all of the kept mass (scored by the whole block from the vector
form), rows of equal values, rows of thousands of kept keys with close scores,
rows longer than 8,192 keys (the two-blocks-per-SM form)."""
import numpy as np
import pytest

from tests.test_gpu_long import check_swap_long, fw  # noqa: F401  (fw is a fixture)
from tests.test_gpu_small import rows_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,v_dtype,E,sink", [(33, 32, "f32", 1, 4), (200, 64, "bf16", 12, 9), (257, 128, "bf16", 40, 8),
                                                (500, 64, "f32", 96, 10), (300, 256, "bf16", 33, 9),
                                                (9001, 64, "bf16", 31, 12)])
def test_swap_extras_and_sinks(fw, n, d, v_dtype, E, sink):  # noqa: F811
    rng = np.random.default_rng(n + E)
    rows = 6
    L = (rng.normal(size=(rows, n)) * rng.uniform(0.3, 2, size=(rows, 1))).astype(np.float32)
    L[:, 0] += sink
    V = rng.normal(size=(rows, n, d)).astype(np.float32)
    k = np.tile(np.array([2, max(2, n // 10), n - 1], np.int32), (rows, 1))
    check_swap_long(fw, rows_batch(L, V, k, v_dtype=v_dtype), E=E, max_swaps=12)


def test_swap_equal_values_take_nothing(fw):  # noqa: F811
    # every set has the same output: no swap strictly lowers es beyond rounding
    import torch

    rng = np.random.default_rng(1)
    L = rng.normal(size=(2, 100)).astype(np.float32)
    V = np.ones((2, 100, 64), np.float32)
    b = rows_batch(L, V, np.full((2, 1), 10))
    rows = fw.rows_from_batch(b)
    k = torch.as_tensor(np.asarray(b.k)).cuda()
    top = fw.dense_and_topk_gap(rows, k)
    sw = fw.swap_refine(rows, k, top, E=32, max_swaps=16)
    torch.cuda.synchronize()
    assert torch.all(sw["refined_gap"] <= sw["topk_gap"] * (1 + 1e-6) + 1e-7)
    assert torch.all(torch.isfinite(sw["refined_gap"]))


@pytest.mark.parametrize("n,k,d,E", [(4000, 2000, 64, 32), (3000, 2900, 128, 96), (700, 350, 256, 40)])
def test_swap_many_kept_keys(fw, n, k, d, E):  # noqa: F811
    # flat rows: thousands of kept keys whose scores lie close together, so the least
    # score keeps falling while the warps use it to leave keys out; the chain is the
    # oracle's whatever moment each warp saw (gaps to the oracle's tolerance: the
    # band sums are added by atomics, in an order that differs from run to run)
    rng = np.random.default_rng(n)
    rows = 4
    L = (0.2 * rng.normal(size=(rows, n))).astype(np.float32)
    V = rng.normal(size=(rows, n, d)).astype(np.float32)
    b = rows_batch(L, V, np.full((rows, 1), k), v_dtype="bf16")
    for _ in range(2):
        check_swap_long(fw, b, E=E, max_swaps=24)
