"""The window scan at the block shapes that a large batch gets by default and a caller cannot ask for: 128 threads
(1,024-slot windows), 224 (8,192), 256 (11,000) and 384 (16,384), each at term counts around one table of that many
terms and at segment lengths around the 8-posting groups and 32-group chunks; and the sampled cut in those shapes (needs
a GB300). Batches have enough blocks for the shape on any device of up to 152 SMs.

All values are whole numbers, so every score is exact in either window: answers are compared exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, never run there
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2509_08395_gb300 as sindi  # noqa: E402
from test_gpu_scan import LENGTHS, _pattern  # noqa: E402

DEV = torch.device("cuda:0")
DIM, NQ, K = 1300, 330, 40
TERMS = [1, 2, 26, 31, 32, 33, 127, 128, 129, 223, 224, 225, 255, 256, 257, 383, 384, 385, 511, 512, 513, 1023, 1024, 1025,
         1300]


def _best(score, k):
    n = score.shape[1]
    key = score.astype(np.int64) * n + (n - 1 - np.arange(n))  # distinct: score descending, then id
    top = -np.sort(-np.partition(key, n - k, axis=1)[:, n - k:], axis=1)
    return n - 1 - top % n, (top // n).astype(np.float32)


@pytest.mark.parametrize("window", [1024, 8192, 11_000, 16_384])
def test_table_edges_in_every_default_shape(window):
    rng = np.random.default_rng(window)
    n = 2 * window + window // 2 + 3
    terms, docs = [], []
    for w in range(3):
        size = min(window, n - w * window)
        for j in range(DIM):
            m = min(LENGTHS[(j + 5 * w) % len(LENGTHS)], size)
            terms.append(np.full(m, j))
            docs.append(w * window + rng.choice(size, m, replace=False))
    term, doc = np.concatenate(terms), np.concatenate(docs)
    order = np.lexsort((term, doc))
    doc, term = doc[order], term[order].astype(np.int32)
    v = rng.integers(1, 5, len(doc)).astype(np.float32)
    ip = np.concatenate([[0], np.cumsum(np.bincount(doc, minlength=n))]).astype(np.int64)
    X = np.zeros((n, DIM))
    X[doc, term] = v
    counts = [TERMS[i % len(TERMS)] for i in range(NQ)]
    picks = [np.sort(rng.choice(DIM, m, replace=False)) for m in counts]
    qp = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    qx = np.concatenate(picks).astype(np.int32)
    qv = rng.integers(1, 5, len(qx)).astype(np.float32)
    Q = np.zeros((NQ, DIM))
    Q[np.repeat(np.arange(NQ), counts), qx] = qv
    ids, top = _best(Q @ X.T, K)
    t = [torch.from_numpy(a).to(DEV) for a in (ip, term, v, qp, qx, qv)]
    with sindi.Index(*t[:3], DIM, window=window) as idx:
        for block in (0, 512):
            for accum in ("f32", "fixed32"):
                for gamma in (0, 200):
                    got, sc = idx.search(*t[3:], k=K, gamma=gamma, mode="batched", block=block, accum=accum)
                    idx.check()
                    np.testing.assert_array_equal(sc.cpu().numpy(), top, err_msg=f"{block} {accum} {gamma}")
                    np.testing.assert_array_equal(got.cpu().numpy(), ids, err_msg=f"{block} {accum} {gamma}")


@pytest.mark.parametrize("window", [1024, 8192, 11_000, 16_384])
@pytest.mark.parametrize("kind", ["outside-the-sample", "inside-the-sample", "ascending", "ties", "few-values", "rare"])
def test_sampled_cuts_in_every_default_shape(kind, window):
    n, nq = 40_000, 400
    v = _pattern(kind, n, np.random.default_rng(window))
    has = v > 0
    ip = np.concatenate([[0], np.cumsum(has)]).astype(np.int64)
    t = [torch.from_numpy(a).to(DEV) for a in (ip, np.zeros(int(ip[-1]), np.int32), v[has].astype(np.float32))]
    w = np.resize(np.array([1.0, 2.0, 0.5], np.float32), nq)
    q = [torch.from_numpy(a).to(DEV) for a in (np.arange(nq + 1, dtype=np.int64), np.zeros(nq, np.int32), w)]
    best = np.lexsort((np.arange(n), -v))  # score descending, then id
    with sindi.Index(*t, 1, window=window) as idx:
        for k, gamma in ((1, 0), (10, 0), (600, 0), (10, 100), (1000, 3000)):
            ids, sc = idx.search(*q, k=k, gamma=gamma, mode="batched")
            idx.check()
            np.testing.assert_array_equal(ids.cpu().numpy(), np.tile(best[:k], (nq, 1)), err_msg=f"{k} {gamma}")
            np.testing.assert_array_equal(sc.cpu().numpy(), (w[:, None] * v[best[:k]][None]).astype(np.float32))
