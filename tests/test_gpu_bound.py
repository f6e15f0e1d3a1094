"""The running bound over scores that are sums of many similar products (binary and small whole values), over scores
with many exact ties, and over answers that reach far below zero (needs a GB300).

All values are whole numbers, so every score is exact in either window and the answer is compared exactly. Windows and
batch sizes are chosen so that the default shapes are blocks of 128 (1,024 slots), 224 (8,192) and 384 threads
(16,384); asked-for shapes run too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, never run there
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2509_08395_gb300 as sindi  # noqa: E402

DEV = torch.device("cuda:0")
N, DIM, NQ, K = 20_000, 300, 240, 60


def _rows(rng, n, nnz, values):
    x = np.sort(np.argsort(rng.random((n, DIM)), axis=1)[:, :nnz], axis=1).astype(np.int32)
    v = values(rng, (n, nnz)).astype(np.float32)
    dense = np.zeros((n, DIM))
    np.put_along_axis(dense, x.astype(np.int64), v, 1)
    return (np.arange(0, n * nnz + 1, nnz, dtype=np.int64), x.ravel(), v.ravel()), dense


KINDS = {  # document values, query values
    "binary": (lambda r, s: np.ones(s), lambda r, s: np.ones(s)),
    "small": (lambda r, s: r.integers(1, 5, s), lambda r, s: r.integers(1, 5, s)),
    "below-zero": (lambda r, s: r.integers(1, 5, s), lambda r, s: -r.integers(1, 5, s)),
    "signed": (lambda r, s: r.integers(1, 5, s) * r.choice([-1, 1], s), lambda r, s: r.integers(1, 5, s)),
}


@pytest.fixture(scope="module", params=[(kind, terms) for kind in KINDS for terms in (20, 100)],
                ids=lambda p: f"{p[0]}-{p[1]}")
def data(request):
    kind, terms = request.param
    rng = np.random.default_rng(terms)
    docs, X = _rows(rng, N, 60, KINDS[kind][0])
    q, Q = _rows(rng, NQ, terms, KINDS[kind][1])
    score = Q @ X.T
    best = np.stack([np.lexsort((np.arange(N), -s))[:K] for s in score])  # score descending, then id
    return [torch.from_numpy(a).to(DEV) for a in (*docs, *q)], best, np.take_along_axis(score, best, 1).astype(np.float32)


@pytest.mark.parametrize("window", [1024, 8192, 16384])
def test_answers_are_exact(data, window):
    t, best, top = data
    with sindi.Index(*t[:3], DIM, window=window) as idx:
        for mode, kw in [(m, dict(block=b, accum=a)) for m in ("plain", "batched") for b in (0, 256, 1024)
                         for a in ("f32", "fixed32")] + [("plain", dict(block=1)), ("batched", dict(block=1)),
                                                         ("batched", dict(group=4))]:
            for gamma in (0, 500):
                ids, sc = idx.search(*t[3:], k=K, gamma=gamma, mode=mode, **kw)
                idx.check()
                np.testing.assert_array_equal(ids.cpu().numpy(), best, err_msg=f"{mode} {kw} {gamma}")
                np.testing.assert_array_equal(sc.cpu().numpy(), top, err_msg=f"{mode} {kw} {gamma}")
