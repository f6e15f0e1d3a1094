"""The device's document pruning at the row lengths, orders and value patterns where its paths change, against the
FP64 oracle's lists (needs a GB300). Counts, ids and FP32 values are equal bit for bit."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, never run there
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2509_08395_gb300 as sindi  # noqa: E402

DEV = torch.device("cuda:0")
DIM = 3000
LENGTHS = [0, 1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2100]


def _values(kind, n, rng):
    if kind == "lognormal":
        return np.exp(0.8 * rng.standard_normal(n)).astype(np.float32)
    if kind == "ties":  # few magnitudes, both signs, explicit zeros
        return (rng.integers(-4, 5, n) / 4).astype(np.float32)
    if kind == "spread":  # magnitudes over the whole FP32 range: FP64 sums round, subnormals included
        return (rng.choice([-1.0, 1.0], n) * np.exp2(rng.uniform(-149.0, 127.0, n))).astype(np.float32)
    assert kind == "edge"  # sums just inside and just outside of 53 bits
    return (1.0 + rng.integers(0, 1 << 23, n) * 2.0 ** -23).astype(np.float32) * np.exp2(
        rng.integers(0, 24, n)).astype(np.float32)


def _rows(kind, shuffled, seed):
    rng = np.random.default_rng(seed)
    lengths = np.array(LENGTHS * 6)
    ip = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    dims = [np.sort(rng.choice(DIM, m, replace=False)) for m in lengths]
    if shuffled:
        dims = [rng.permutation(d) if i % 2 else d for i, d in enumerate(dims)]
    return ip, np.concatenate(dims).astype(np.int32), _values(kind, int(ip[-1]), rng)


def _by_id(ex):
    seg = ex["seg"].astype(np.int64)
    of = np.repeat(np.arange(len(seg) - 1), np.diff(seg))
    order = np.lexsort((ex["ids"], of))
    return ex["ids"][order].astype(np.int64), ex["vals"][order]


@pytest.mark.parametrize("kind", ["lognormal", "ties", "spread", "edge"])
@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("prune,alpha,vn", [("mass", 0.5, 0), ("mass", 1e-9, 0), ("mass", 0.999, 0), ("mass", 1.0, 0),
                                            ("vector_number", 1.0, 33), ("vector_number", 1.0, 1)])
def test_pruned_rows_equal_the_oracles(kind, shuffled, prune, alpha, vn):
    ip, ix, v = _rows(kind, shuffled, seed=7 + len(kind) + 2 * shuffled)
    I = oracle.Index(oracle.Dataset(ip, ix, v, DIM), window=50, alpha=alpha, prune=prune, prune_n=vn)
    seg, pid, pval, _, kept = I.export()
    t = [torch.from_numpy(a).to(DEV) for a in (ip, ix, v)]
    with sindi.Index(*t, DIM, window=50, alpha=alpha, prune=prune, prune_n=vn) as idx:
        ex = idx.export()
    np.testing.assert_array_equal(ex["kept"].astype(np.int64), kept)
    np.testing.assert_array_equal(ex["seg"].astype(np.int64), seg)
    ids, vals = _by_id(ex)
    np.testing.assert_array_equal(ids, pid % 50)
    np.testing.assert_array_equal(vals, pval.astype(np.float32))


@pytest.mark.parametrize("length", [5, 64, 300, 700, 1500])
@pytest.mark.parametrize("fault,text", [("dim", "outside"), ("dup", "repeated"), ("inf", "non-finite"),
                                        ("nan", "non-finite")])
def test_a_malformed_row_is_refused_on_every_path(length, fault, text):
    rng = np.random.default_rng(length)
    ip = np.arange(0, 21 * length, length, dtype=np.int64)
    ix = np.concatenate([np.sort(rng.choice(DIM, length, replace=False)) for _ in range(20)]).astype(np.int32)
    v = np.ones(20 * length, np.float32)
    at = 13 * length + length - 1
    if fault == "dim":
        ix[at] = DIM
    elif fault == "dup":
        ix[at] = ix[13 * length]
    else:
        v[at] = np.inf if fault == "inf" else np.nan
    with pytest.raises(sindi.SindiError, match=text):
        sindi.Index(*[torch.from_numpy(a).to(DEV) for a in (ip, ix, v)], DIM, window=50, alpha=0.5)
