"""List pruning where one list holds much of the collection (ranked by a sort) and where none does (selected by a block
a list), against the FP64 oracle's lists (needs a GB300). Counts, ids and FP32 values are equal bit for bit."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, never run there
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2509_08395_gb300 as sindi  # noqa: E402

DEV = torch.device("cuda:0")
N = 3000


def _docs(dim, most, values, seed):
    rng = np.random.default_rng(seed)
    dims = [np.sort(rng.choice(dim, rng.integers(0, min(dim, most) + 1), replace=False)) for _ in range(N)]
    ip = np.concatenate([[0], np.cumsum([len(d) for d in dims])]).astype(np.int64)
    n = int(ip[-1])
    v = {"lognormal": lambda: np.exp(0.8 * rng.standard_normal(n)), "ties": lambda: rng.integers(-3, 4, n) / 4,
         "one-value": lambda: np.ones(n)}[values]()
    return ip, np.concatenate(dims).astype(np.int32), v.astype(np.float32)


def _by_id(ex):
    seg = ex["seg"].astype(np.int64)
    of = np.repeat(np.arange(len(seg) - 1), np.diff(seg))
    order = np.lexsort((ex["ids"], of))
    return ex["ids"][order].astype(np.int64), ex["vals"][order]


# dims 1 .. 70 are sorted (the longest list is more than 1/90 of the postings), 700 dims selected
@pytest.mark.parametrize("values", ["lognormal", "ties", "one-value"])
@pytest.mark.parametrize("dim,most", [(1, 1), (2, 2), (17, 6), (70, 20), (700, 20)])
@pytest.mark.parametrize("prune,lp,alpha", [("list", 1, 1.0), ("list", 37, 1.0), ("list", 1500, 1.0), ("list", 10_000, 1.0),
                                            ("mass_list", 30, 0.6)])
def test_pruned_lists_equal_the_oracles(dim, most, values, prune, lp, alpha):
    ip, ix, v = _docs(dim, most, values, seed=dim)
    I = oracle.Index(oracle.Dataset(ip, ix, v, dim), window=700, alpha=alpha, prune=prune, prune_n=lp)
    seg, pid, pval, _, kept = I.export()
    t = [torch.from_numpy(a).to(DEV) for a in (ip, ix, v)]
    with sindi.Index(*t, dim, window=700, alpha=alpha, prune=prune, prune_n=lp) as idx:
        ex = idx.export()
    np.testing.assert_array_equal(ex["kept"].astype(np.int64), kept)
    np.testing.assert_array_equal(ex["seg"].astype(np.int64), seg)
    ids, vals = _by_id(ex)
    np.testing.assert_array_equal(ids, pid % 700)
    np.testing.assert_array_equal(vals, pval.astype(np.float32))
