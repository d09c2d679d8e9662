"""The three-point check of linearly scanned items: a warp per item on short
lists, four lanes per item on longer ones.

Route 1 sends every item to the linear FP32 scan and its check, so the list is
the batch: sizes around the grid's 2,432 warps, where the form changes, and
models around the 8 layers that a point's lanes take at a time. Indices are
whole numbers: equal to the FP64 scan's.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2003_02256_gb300 import masw  # noqa: E402
from paper_2003_02256_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("n_items", [1, 3, 2432, 2433])
@pytest.mark.parametrize("layers", [0, 1, 7, 8, 9, 17])
def test_checked_items_equal_the_fp64_scan(n_items, layers):
    if layers:
        m, g = W.ragged_batch(1, layers=(layers, layers), lambdas=(n_items, n_items),
                              invert_frac=1.0 if layers > 1 else 0.0, seed=layers)
    else:
        _, g = W.ragged_batch(1, seed=1)
        m = W.Models(np.zeros(1, np.int32), np.zeros(0), np.array([700.0]), np.array([400.0]),
                     np.array([1900.0]), np.array([n_items], np.int32),
                     np.geomspace(1.0, 200.0, n_items))
    with masw.Batch(m, g) as b:
        b.set_plan(precision=0)
        want = b.dispersion()[1]
        b.set_plan(precision=2)
        b.set_route(1)
        got = b.dispersion()[1]
    assert np.array_equal(want, got)
