"""sindi_release_memory without a GPU: argument checks only."""
import pytest

import paper_2509_08395_gb300 as sindi
from paper_2509_08395_gb300 import build_native


@pytest.mark.parametrize("device", [-1, 10_000])
def test_a_device_that_does_not_exist_is_refused(device):
    build_native.build()
    with pytest.raises(sindi.SindiError, match="no such device"):
        sindi.sindi_release_memory(device)
