"""Batch plans at the edges of what sorts and ranks the tokens: warps, the sort's widths, chunks of 256."""
import numpy as np
import pytest

from test_gpu_plan import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 31, 32, 33, 127, 128, 129, 255, 257, 511, 513, 1023, 1024, 1025, 1055, 1057, 1280, 1281, 4000])
@pytest.mark.parametrize("E", [1, 5, 700])
def test_sizes(T, E):
    rng = np.random.default_rng(T * 1000 + E)
    _check(rng.integers(-1, E, size=T).astype(np.int32), E)
