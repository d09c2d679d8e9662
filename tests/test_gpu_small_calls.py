"""Small calls: results of a batch in one host copy, gradient index tensors
laid out once per batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2003_02256_gb300 import autograd, masw  # noqa: E402
from paper_2003_02256_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("n_items", [1, 2, 4095, 4096, 4097])
@pytest.mark.parametrize("kinds", [("host",) * 3, ("pinned",) * 3, ("host", "device", "pinned")])
def test_host_results_equal_device_results(n_items, kinds):
    m, g = W.ragged_batch(1, layers=(3, 3), lambdas=(n_items, n_items), seed=5)

    def buffer(kind, dtype):
        if kind == "host":
            return np.full(n_items, -7, dtype=dtype)
        t = torch.full((n_items,), -7, dtype=torch.float64 if dtype == np.float64 else torch.int32)
        return t.cuda() if kind == "device" else t.pin_memory()

    dtypes = (np.float64, np.int32, np.int32)
    with masw.Batch(m, g) as b:
        want = [buffer("device", d) for d in dtypes]
        got = [buffer(k, d) for k, d in zip(kinds, dtypes)]
        masw.dispersion(b.handle, *want)
        masw.dispersion(b.handle, *got)
        ce = np.full(n_items, 300.0)
        phi = np.empty(1)
        got2 = [buffer(k, d) for k, d in zip(kinds, dtypes)]
        masw.misfit_curves(b.handle, ce, masw.MISFIT_LSQ, 2.0, phi, *got2)
        torch.cuda.synchronize()
        for w, *rest in zip(want, got, got2):
            for a in rest:
                assert np.array_equal(w.cpu().numpy(), np.asarray(a.cpu() if torch.is_tensor(a) else a),
                                      equal_nan=True)


def test_gradient_after_a_pass_in_inference_mode():
    m, g, _ = W.differentiation_batch(n_models=3, n_lambda=10)
    ce = np.full(m.n_items, 300.0)
    grads = []
    for first in (False, True):
        with masw.Batch(m, g) as b:
            beta = torch.tensor(m.beta, device="cuda", requires_grad=True)
            h = torch.tensor(m.h, device="cuda", requires_grad=True)
            if first:
                with torch.inference_mode():
                    autograd.misfit(beta, h, b, ce)
            phi = autograd.misfit(beta, h, b, ce)
        phi.sum().backward()
        grads.append((beta.grad, h.grad))
    assert torch.equal(grads[0][0], grads[1][0]) and torch.equal(grads[0][1], grads[1][1])
