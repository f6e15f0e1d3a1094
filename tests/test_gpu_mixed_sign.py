"""Queries with negative values over documents without any: zero scores rank above negative ones, so a window may not
leave its zero-score slots out, wherever in the query the negative values stand (needs a GB300).

Values are whole numbers: every score is exact in either window, and the answer is compared exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, never run there
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2509_08395_gb300 as sindi  # noqa: E402

DEV = torch.device("cuda:0")
N, DIM, K = 20_000, 2_000, 300
NEG = 1_990  # the documents' other dims: NEG .. NEG + 7; DIM - 1 is in no query


@pytest.fixture(scope="module")
def docs():
    """One entry a document: 100 documents score above zero, 60 at zero, the others below, in random places."""
    rng = np.random.default_rng(2)
    kind = rng.permutation(np.repeat([0, 1, 2], [100, 60, N - 160]))
    j = np.select([kind == 0, kind == 1], [rng.integers(0, 32, N), DIM - 1], NEG + rng.integers(0, 8, N))
    return np.arange(N + 1, dtype=np.int64), j.astype(np.int32), rng.integers(1, 50, N).astype(np.float32)


@pytest.mark.parametrize("window", [1024, 4096])
@pytest.mark.parametrize("accum", ["f32", "fixed32"])
@pytest.mark.parametrize("block", [0, 256, 1024])
@pytest.mark.parametrize("terms", [33, 40, 64, 257, 1032])
def test_negative_values_late_in_the_query(docs, terms, block, accum, window):
    """The negative values are the query's last (from its 33rd entry on at the earliest): one to eight of them."""
    n_neg = min(8, terms - 32)
    qx = np.concatenate([np.arange(terms - n_neg), NEG + np.arange(n_neg)]).astype(np.int32)
    qv = np.where(np.arange(terms) < terms - n_neg, 3.0, -2.0).astype(np.float32)
    w = np.zeros(DIM)
    w[qx] = qv
    score = w[docs[1]] * docs[2]
    best = np.lexsort((np.arange(N), -score))[:K]  # score descending, then id
    nq = 40
    q = (np.arange(0, nq * terms + 1, terms, dtype=np.int64), np.tile(qx, nq), np.tile(qv, nq))
    t = [torch.from_numpy(a).to(DEV) for a in (*docs, *q)]
    with sindi.Index(*t[:3], DIM, window=window) as idx:
        for mode in ("plain", "batched"):
            for gamma in (0, 350):
                ids, sc = idx.search(*t[3:], k=K, gamma=gamma, mode=mode, block=block, accum=accum)
                idx.check()
                np.testing.assert_array_equal(ids.cpu().numpy(), np.tile(best, (nq, 1)), err_msg=f"{mode} {gamma}")
                np.testing.assert_array_equal(sc.cpu().numpy(), np.tile(score[best].astype(np.float32), (nq, 1)))
