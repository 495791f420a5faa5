"""The long-row select at the lengths where its thread layout changes and on
rows that leave the linear bins: kept bits, thresholds and softmax statistics
against plain numpy, including NaN and infinite logits and ranges fp32 cannot
scale."""
import ctypes

import numpy as np
import pytest

from tests.parity import np_
from tests.test_gpu_small import rows_batch

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fw():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_25230_gb300 import fw as _fw

    return _fw


def kept(l, k):
    m = np.zeros(len(l), bool)
    m[np.lexsort((np.arange(len(l)), -l.astype(np.float64)))[:k]] = True
    return m


def run(fw, L, ks):
    rows, n = L.shape
    V = np.ones((rows, n, 32), np.float32)
    b = rows_batch(L, V, np.tile(np.asarray(ks, np.int32), (rows, 1)))
    g = fw.dense_and_topk_gap(fw.rows_from_batch(b), torch.as_tensor(np.asarray(b.k)).cuda())
    torch.cuda.synchronize()
    return {k: np_(v) for k, v in g.items() if not k.startswith("_")}


def check(g, r, l, ks):
    n = len(l)
    assert g["row_status"][r] == 0
    for b, k in enumerate(ks):
        w = g["kept_bits"][r, b].view(np.uint32)
        bits = ((w[np.arange(len(w) * 32) >> 5] >> (np.arange(len(w) * 32) & 31)) & 1).astype(bool)
        assert not bits[n:].any()
        np.testing.assert_array_equal(bits[:n], kept(l, k))
    p = np.exp(l.astype(np.float64) - l.max())
    assert g["row_max"][r] == l.max() and abs(g["row_sum"][r] - p.sum()) <= 1e-5 * p.sum()


@pytest.mark.parametrize("n", [33, 63, 1023, 1024, 1025, 2049, 4095, 4097, 8193, 16383, 16385, 32767, 32768])
def test_select_lengths(fw, n):
    rng = np.random.default_rng(n)
    L = (rng.normal(size=(5, n)) * rng.uniform(0.2, 5, size=(5, 1))).astype(np.float32)
    L[1, :] = np.round(L[1] * 4) / 4      # ties
    L[2, : n // 2] = -0.0                 # signed zeros
    L[2, n // 2:] = 0.0
    L[3] += 1e6                           # a small range far from 0
    L[4, 0] = 1e4                         # one key far above the rest: crowded bins
    ks = [1, max(1, n // 16), n // 2, n]
    for nb in (1, 3, 4):
        g = run(fw, L, ks[-nb:])
        for r in range(5):
            check(g, r, L[r], ks[-nb:])


def test_select_nonfinite_and_wide_rows(fw):
    rng = np.random.default_rng(0)
    L = rng.normal(size=(6, 5000)).astype(np.float32)
    L[0, 4321] = np.nan
    L[1, 17] = np.inf
    L[2, 18] = -np.inf
    L[3, 5], L[3, 6] = 3e38, -3e38        # a range that overflows
    L[4] *= 1e37
    g = run(fw, L, [7, 2500])
    assert list(g["row_status"][:3]) == [fw.FW_ERR_NONFINITE] * 3
    for r in (3, 4, 5):
        check(g, r, L[r], [7, 2500])


@pytest.mark.parametrize("n,words", [(33, 2), (1000, 40), (1024, 33), (5000, 1500), (20, 9)])
def test_select_writes_every_word(fw, n, words):
    # more words than the row has: zero past its keys, on rows that stay in the linear
    # bins and on one that goes to the radix select
    rng = np.random.default_rng(n)
    L = rng.normal(size=(3, n)).astype(np.float32)
    L[1, :3] = 3e38, -3e38, 0
    b = rows_batch(L, np.ones((3, n, 32), np.float32), np.tile(np.array([1, n // 2], np.int32), (3, 1)))
    rows, k = fw.rows_from_batch(b), torch.as_tensor(np.asarray(b.k)).cuda()
    top = fw.dense_and_topk_gap(rows, k)
    bits = torch.full((3 * 2 * words + 64,), -1, dtype=torch.int32, device="cuda")
    c = top["_c"]
    c.kept_bits, c.kept_words = bits.data_ptr(), words
    ws = torch.empty(fw.raw().fw_dense_and_topk_gap_workspace(ctypes.byref(rows.c), 2) + 256, dtype=torch.uint8, device="cuda")
    assert fw.raw().fw_dense_and_topk_gap(ctypes.byref(rows.c), fw._ptr(k), 2, ctypes.byref(c), fw._ptr(ws), ws.numel(),
                                          fw._stream(None)) == 0
    torch.cuda.synchronize()
    assert (bits[-64:] == -1).all()
    w = np_(bits[:-64]).view(np.uint32).reshape(3, 2, words)
    for r in range(3):
        check(dict(row_status=np.zeros(3), kept_bits=w, row_max=L.max(1), row_sum=np_(top["row_sum"])), r, L[r], [1, n // 2])
