"""The counting plans' proofs: FP32 counts with an error bound, completed in
double-float where the bound decides nothing.

Every form of the plan reports the pure FP64 scan's index for every item, at
the sizes where the lists, passes and lane assignments of its kernels have
edges: single items, a model shorter than the anchor stride, counts around a
warp and a block, a half-space alone, models whose first change lies above the
pole-free range or below the first test velocity, and thin layers at long
wavelengths, where the FP32 recurrence carries its largest relative errors.
Indices are whole numbers: the comparison is exact.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2003_02256_gb300 import masw  # noqa: E402
from paper_2003_02256_gb300 import workloads as W  # noqa: E402


def _edge_models(seed):
    """Ragged models with 0..30 layers and 1, 2, 6, 7, 13, ... wavelengths."""
    rng = np.random.default_rng(seed)
    parts = []
    for n_lambda in (1, 2, 5, 6, 7, 8, 12, 13, 31, 32, 33, 64, 65):
        m, _ = W.ragged_batch(1, layers=(0, 30) if n_lambda == 1 else (1, 30),
                              lambdas=(n_lambda, n_lambda), invert_frac=0.5,
                              seed=int(rng.integers(1 << 30)))
        m.lam[:] = np.geomspace(1.0, 200.0, n_lambda)
        parts.append(m)
    half = W.Models(np.zeros(1, np.int32), np.zeros(0), np.array([700.0]), np.array([400.0]),
                    np.array([1900.0]), np.array([3], np.int32), np.array([1.0, 30.0, 900.0]))
    return W.concat(parts + [half])


def _thin_models(seed):
    """Layers of 5 cm .. 1 m at wavelengths up to 500 m."""
    m, _ = W.extreme_batch(24, n_lambda=21, seed=seed)
    rng = np.random.default_rng(seed)
    m.h[:] = np.exp(rng.uniform(np.log(0.05), 0.0, m.h.size))
    m.lam[:] = np.tile(np.geomspace(0.5, 500.0, 21), 24)
    return m


CASES = {
    "edges": (lambda: _edge_models(3), W.Grid(50.0, 0.25, 4601)),
    "grid starts above modes": (lambda: _edge_models(4), W.Grid(300.0, 0.7, 1201)),
    "thin layers": (lambda: _thin_models(5), W.Grid(50.0, 0.5, 2901)),
    "extreme": (lambda: W.extreme_batch(64, seed=6)[0], W.Grid(50.0, 0.5, 4901)),
    "one item": (lambda: W.uniform_batch(1, 3, 1, seed=7)[0], W.Grid(50.0, 0.25, 4601)),
    "two grid points": (lambda: W.uniform_batch(3, 2, 129, seed=8)[0], W.Grid(200.0, 30.0, 2)),
}


@pytest.mark.parametrize("name", CASES)
def test_counting_forms_equal_the_fp64_scan(name):
    make, grid = CASES[name]
    models = make()
    with masw.Batch(models, grid) as b:
        b.set_plan(precision=0)
        ct0, idx0, st0 = b.dispersion()
        for split in (0, 1, 2):
            for block in (64, 128, 256):
                b.set_plan(precision=2, count_split=split, count_block=block)
                for _ in range(2):  # the second pass over the same lists and counters
                    ct, idx, st = b.dispersion()
                    assert np.array_equal(idx, idx0), (split, block, np.flatnonzero(idx != idx0))
                    assert np.array_equal(st, st0)
                    assert np.array_equal(ct, ct0, equal_nan=True)
