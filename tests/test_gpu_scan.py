"""The window scan's group table at its edges (segment lengths around the 8-posting groups and 32-group chunks, empty
lists, queries around one term table), against the scores in 64 bits (needs a GB300).

Tolerances: the values are positive, so a score of m <= 700 FP32 products is within (m + 1) * 2^-24 < 4.2e-5 relative
of the exact one; the fixed-point window adds m * B * 2^-30 (B: the sum of the terms' largest products), at most
m * 2^-30 * B / score, below 6.6e-5 for scores above B / 100. Scores here are compared at 1.1e-4."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, never run there
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2509_08395_gb300 as sindi  # noqa: E402

DEV = torch.device("cuda:0")
TOL = 1.1e-4
N, LAMBDA = 2600, 1024  # windows of 1,024, 1,024 and 552 documents
LENGTHS = [0, 1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 250, 255, 256, 257, 264, 511, 513, 552]


def _lists(n_terms, seed):
    """CSR documents in which term j has LENGTHS[(j + 5 w) mod len] postings in window w."""
    rng = np.random.default_rng(seed)
    rows = [[] for _ in range(N)]
    for j in range(n_terms):
        for w in range(3):
            size = min(LAMBDA, N - w * LAMBDA)
            for m in rng.choice(size, LENGTHS[(j + 5 * w) % len(LENGTHS)], replace=False):
                rows[w * LAMBDA + m].append((j, rng.uniform(0.5, 2.0)))
    ip = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    ix = np.array([j for r in rows for j, _ in r], np.int32)
    v = np.array([x for r in rows for _, x in r], np.float32)
    X = np.zeros((N, n_terms))
    X[np.repeat(np.arange(N), np.diff(ip)), ix] = v
    return ip, ix, v, X


@pytest.mark.parametrize("accum", ["f32", "fixed32"])
@pytest.mark.parametrize("block", [0, 256, 1024])
@pytest.mark.parametrize("n_terms", [26, 78, 255, 257, 520, 700])
def test_group_table_edges(n_terms, block, accum):
    ip, ix, v, X = _lists(n_terms, seed=n_terms)
    rng = np.random.default_rng(1)
    # every term; one term of each length alone; random subsets (among them terms that are empty in a window)
    picks = [np.arange(n_terms)] + [np.array([j]) for j in range(26)] + [
        np.sort(rng.choice(n_terms, rng.integers(2, n_terms), replace=False)) for _ in range(9)]
    qp = np.concatenate([[0], np.cumsum([len(p) for p in picks])]).astype(np.int64)
    qx = np.concatenate(picks).astype(np.int32)
    qv = rng.uniform(0.5, 2.0, len(qx)).astype(np.float32)
    t = [torch.from_numpy(a).to(DEV) for a in (ip, ix, v, qp, qx, qv)]
    k = 40
    with sindi.Index(*t[:3], n_terms, window=LAMBDA) as idx:
        out = {}
        for mode in ("plain", "batched"):
            ids, sc = idx.search(*t[3:], k=k, mode=mode, block=block, accum=accum)
            idx.check()
            out[mode] = ids.cpu().numpy().astype(np.int64), sc.cpu().numpy()
    for mode, (ids, sc) in out.items():
        for r, p in enumerate(picks):
            exact = X[:, p] @ qv[qp[r]:qp[r + 1]].astype(np.float64)
            best = np.sort(exact)[::-1][:k]
            assert len(set(ids[r])) == k
            np.testing.assert_allclose(sc[r], exact[ids[r]], rtol=TOL, atol=0, err_msg=f"{mode} {r}")
            np.testing.assert_allclose(sc[r], best, rtol=TOL, atol=0, err_msg=f"{mode} {r}")


def _pattern(kind, n, rng):
    """One value per document (0: not in the list), whole numbers: every sum below is exact in either window."""
    base = rng.permutation(n).astype(np.int64) + 1
    span = np.arange(n) // 128 % 8
    if kind == "outside-the-sample":  # the best slots lie in spans the sampled cut does not read
        return base + n * (span != 0)
    if kind == "inside-the-sample":
        return base + n * (span == 0)
    if kind == "ascending":
        return np.arange(1, n + 1)
    if kind == "ties":
        return np.full(n, 7)
    if kind == "few-values":
        return base % 3 + 1
    assert kind == "rare"  # fewer scored documents than candidates
    return np.where(rng.random(n) < 0.004, base, 0)


@pytest.mark.parametrize("window", [300, 1024, 16384, 32768])
@pytest.mark.parametrize("kind", ["outside-the-sample", "inside-the-sample", "ascending", "ties", "few-values", "rare"])
def test_sampled_cuts_keep_the_exact_answer(kind, window):
    n = 40_000
    rng = np.random.default_rng(window)
    v = _pattern(kind, n, rng)
    has = v > 0
    ip = np.concatenate([[0], np.cumsum(has)]).astype(np.int64)
    t = [torch.from_numpy(a).to(DEV) for a in (ip, np.zeros(int(ip[-1]), np.int32), v[has].astype(np.float32))]
    nq = 3
    q = [torch.from_numpy(a).to(DEV) for a in (np.arange(nq + 1, dtype=np.int64), np.zeros(nq, np.int32),
                                               np.array([1.0, 2.0, 0.5], np.float32))]
    best = np.lexsort((np.arange(n), -v))  # score descending, then id
    with sindi.Index(*t, 1, window=window) as idx:
        for mode in ("plain", "batched"):
            for k, gamma in ((1, 0), (10, 0), (600, 0), (10, 100), (1000, 3000)):
                ids, sc = idx.search(*q, k=k, gamma=gamma, mode=mode)
                idx.check()
                for r, w in enumerate((1.0, 2.0, 0.5)):
                    np.testing.assert_array_equal(ids[r].cpu().numpy(), best[:k], err_msg=f"{mode} {k} {gamma} {r}")
                    np.testing.assert_array_equal(sc[r].cpu().numpy(), (w * v[best[:k]]).astype(np.float32))
