"""Refined roots of sign changes that are no simple root: poles of det K.

A first change with a count change of -1 is a clamped-layer mode, where the
determinant changes sign through infinity. Its "root" is what regula falsi on
the determinant closes in on, to no better than its slow convergence there, so
it has to come from the grid interval itself; the oracle's bisection of the
same interval is within 1e-9, and simple roots are within 1e-12.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2003_02256_gb300 import masw  # noqa: E402
from paper_2003_02256_gb300 import workloads as W  # noqa: E402


def test_roots_at_poles_and_simple_roots(oracle_lib):
    m, g = W.ragged_batch(600, seed=11)
    with masw.Batch(m, g) as b:
        root = b.roots()
        _, idx, _, delta = b.changes(1)
    idx, delta = idx[:, 0], delta[:, 0]
    owner = np.repeat(np.arange(m.n_models), m.n_lambda)
    pick = np.flatnonzero((idx >= 1) & (delta != 1))
    pick = np.concatenate([pick, np.flatnonzero(delta == 1)[::997]])
    for i in pick:
        h, a, be, rho, _ = m.model(int(owner[i]))
        want = oracle_lib.root(h, a, be, rho, m.lam[i], g.c0, g.dc, g.n_c, int(idx[i]))
        assert abs(root[i] - want) <= (1e-12 if delta[i] == 1 else 1e-9) * want
