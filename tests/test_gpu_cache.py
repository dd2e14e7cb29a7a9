"""The value cache of gsn_eval / gsn_expected beside the other calls that build per-species shapes."""
import numpy as np
import pytest

from oracle import gsn_oracle as O
from paper_1812_05686_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("toys", [1, 5])
def test_values_after_a_rate_fit(precision, toys):
    """A rate fit at another response point leaves the values at the cached point as they were, bit for bit."""
    torch = pytest.importorskip("torch")
    from paper_1812_05686_gb300 import gsn
    w = I.borexino_like(n_bins=70, n_fine=300, e_max=0.2)
    n = np.concatenate([I.poisson_counts(O.expected_counts(w, w["theta0"], d), 3 + d) for d in range(2)])
    ctx = gsn.context_from_workload(w, precision, counts=n)
    th = w["theta0"]
    before = ctx.eval(th)[1], ctx.expected(th, 0), ctx.expected(th, 1)
    dev = torch.device("cuda", 0)
    start = np.repeat(th[None], toys, axis=0)
    start[:, w["spectra"].shape[0]] *= 0.9     # light yield
    free = np.zeros(w["n_params"], bool)
    free[w["slot_map"][0, :2]] = True
    ctx.fit_rates_batch_dev(torch.tensor(start, device=dev), torch.tensor(np.tile(n, (toys, 1)), device=dev),
                            torch.tensor([[[0, 70], [0, 70]]] * toys, dtype=torch.int32, device=dev), free, lo=np.where(free, 0.0, -np.inf))
    after = ctx.eval(th)[1], ctx.expected(th, 0), ctx.expected(th, 1)
    for a, b in zip(before, after):
        assert np.array_equal(a, b)
    ctx.close()
