"""sindi_release_memory: what builds and searches leave in the library's pool goes back to the device, indexes that are
alive keep working (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU machines, never run there
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2509_08395_gb300 as sindi  # noqa: E402

DEV = torch.device("cuda:0")


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info(DEV)[0]


def test_unused_memory_goes_back_and_indexes_stay():
    n, dim, nnz = 400_000, 5_000, 60
    g = torch.Generator(device=DEV)
    g.manual_seed(1)
    ip = torch.arange(0, n * nnz + 1, nnz, device=DEV)
    step = torch.randint(1, dim // nnz, (n, nnz), generator=g, device=DEV)
    ix = (step.cumsum(1) - 1).int().flatten()
    v = torch.rand(n * nnz, generator=g, device=DEV) + 0.5
    q = (ip[:9].clone(), ix[:8 * nnz].clone(), v[:8 * nnz].clone())
    small = sindi.Index(ip[:1001], ix[:1000 * nnz], v[:1000 * nnz], dim, window=1024)
    before = small.search(*q, k=10, gamma=50)
    sindi.sindi_release_memory()
    del step
    base = _free()
    big = sindi.Index(ip, ix, v, dim, window=8192)
    big.search(*q, k=10, gamma=500, mode="batched")
    doc_bytes = big.info["doc_bytes"]
    big.close()
    held = base - _free()
    assert held >= doc_bytes  # the freed index's memory is still the pool's
    sindi.sindi_release_memory()
    assert base - _free() < 64 << 20
    after = small.search(*q, k=10, gamma=50)
    small.check()
    for a, b in zip(before, after):
        np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy())
    small.close()
