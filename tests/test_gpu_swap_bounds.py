"""The long-row swap kernel where its bounds and branches change: extras that do
not fill a lane's eight slots, several blocks of 32 slots, rows whose sink
holds nearly all of the kept mass (scored by the whole block from the vector
form), rows of equal values, rows of thousands of kept keys with close scores,
rows longer than 8,192 keys (the two-blocks-per-SM form)."""
import numpy as np
import pytest

import oracle
from tests.parity import assert_close, np_, row_onorm
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


@pytest.mark.parametrize("value", [0.0, 1.0])
def test_swap_equal_values(fw, value):  # noqa: F811
    # every set has the same output.  Zeros: every score is exactly 0, nothing is taken.
    # Ones: es is rounding noise and swaps may follow it, but they are swaps of kept
    # for dropped keys, and the gap of any set is 0 to the oracle's floor
    import torch

    rng = np.random.default_rng(1)
    L = rng.normal(size=(2, 100)).astype(np.float32)
    V = np.full((2, 100, 64), value, np.float32)
    b = rows_batch(L, V, np.full((2, 1), 10))
    rows = fw.rows_from_batch(b)
    k = torch.as_tensor(np.asarray(b.k)).cuda()
    top = fw.dense_and_topk_gap(rows, k)
    sw = {x: np_(v) for x, v in fw.swap_refine(rows, k, top, E=32, max_swaps=16).items() if not x.startswith("_")}
    if value == 0.0:
        assert not sw["n_swaps"].any() and (sw["swap_out"] == -1).all() and (sw["swap_in"] == -1).all()
        assert not sw["refined_gap"].any() and not sw["topk_gap"].any()
    for r in range(2):
        m = int(sw["n_swaps"][r, 0])
        assert 0 <= m <= 16 and (sw["swap_out"][r, 0, m:] == -1).all() and (sw["swap_in"][r, 0, m:] == -1).all()
        kept = set(np.lexsort((np.arange(100), -L[r].astype(np.float64)))[:10].tolist())
        for i, j in zip(sw["swap_out"][r, 0, :m].tolist(), sw["swap_in"][r, 0, :m].tolist()):
            assert i in kept and j not in kept and 0 <= j < 100
            kept = kept - {i} | {j}
    assert_close(sw["refined_gap"], 0 * sw["refined_gap"], np.full(2, 8.0 * value), "refined_gap")  # ||o|| = 8


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


@pytest.mark.parametrize("n,k,d", [(3000, 1000, 256), (2500, 600, 64), (2000, 500, 32)])
def test_swap_long_chains(fw, n, k, d):  # noqa: F811
    # 80 to 100 swaps a row, to the end of the chain: the decisions are still good (the
    # oracle's near-ties may part the two, but every swap lowers the fp64 gap and the
    # chain ends as low as the oracle's), and the gap is that of the set the swaps name
    import torch

    rng = np.random.default_rng(n)
    rows = 3
    L = (0.5 * rng.normal(size=(rows, n))).astype(np.float32)
    V = rng.normal(size=(rows, n, d))
    V += 0.5 * np.sign(L)[:, :, None] * rng.normal(size=(rows, 1, d))  # top-mass values lean to one side
    V = V.astype(np.float32)
    b = rows_batch(L, V, np.full((rows, 1), k))
    r = fw.rows_from_batch(b)
    kt = torch.as_tensor(np.asarray(b.k)).cuda()
    sw = fw.swap_refine(r, kt, fw.dense_and_topk_gap(r, kt), E=96, max_swaps=400)
    o = oracle.swap_refine(b, E=96, max_swaps=400)
    on = row_onorm(oracle.dense_and_topk_gap(b)["o"])
    assert_close(np_(sw["refined_gap"]), o["refined_gap"], on, "refined_gap")
    assert o["n_swaps"].min() >= 60 and not np_(sw["capped"]).any()
    for row in range(rows):
        l, v = L[row].astype(np.float64), V[row].astype(np.float64)
        p = np.exp(l - l.max())
        p /= p.sum()
        u = p[:, None] * (v - p @ v)
        kept = np.zeros(n, bool)
        kept[np.lexsort((np.arange(n), -l))[:k]] = True
        es = np.linalg.norm(u[kept].sum(0)) / p[kept].sum()
        for i, j in np_(torch.stack([sw["swap_out"][row, 0], sw["swap_in"][row, 0]], 1))[:int(sw["n_swaps"][row, 0])]:
            assert kept[i] and not kept[j]
            kept[i], kept[j] = False, True
            last, es = es, np.linalg.norm(u[kept].sum(0)) / p[kept].sum()
            assert es < last * (1 + 1e-6)  # (fp32 cannot tell smaller steps from none)
        assert abs(float(sw["refined_gap"][row, 0]) - es) <= 1e-4 * es + 1e-6 * on[row]
