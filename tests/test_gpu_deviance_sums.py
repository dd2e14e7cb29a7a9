"""Poisson terms one by one, and sums of very many of them (template fits: the expectation is exact)."""
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_1812_05686_gb300 import inputs as I

pytestmark = pytest.mark.gpu
getcontext().prec = 50


def _term(mu, n):
    mu, n = Decimal(float(mu)), Decimal(float(n))
    return mu - n + (n * (n / mu).ln() if n > 0 else 0)


def _flat(J, D):
    w = I.template_like(n_bins=J, n_species=1)
    rep = lambda v: np.repeat(np.asarray(v)[:1], D, axis=0)
    return dict(w, edges=[w["edges"][0]] * D, exposure=np.ones(D), mask=np.repeat(w["mask"][:, :1], D, axis=1),
                slot_map=rep(w["slot_map"]), win_lo=rep(w["win_lo"]), win_hi=rep(w["win_hi"]), templates=[[np.ones(J)] * D])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [1, 7, 1000, 10**7])
def test_single_terms(n, precision):
    """One bin, expectations at ratios inside the series' range (0.667 .. 1.5): the term relative to itself, six
    operations of 2^-46 each; outside it, the logarithm's rounding against the count."""
    from paper_1812_05686_gb300 import gsn
    ctx = gsn.context_from_workload(_flat(1, 1), precision, counts=np.array([float(n)]))
    for r in (0.67, 0.7, 0.9, 0.99, 0.9999, 1.0001, 1.02, 1.2, 1.4, 1.49):
        rc, nll, _ = ctx.eval_grad(np.array([n / r]))
        assert rc == 0, ctx.last_error()
        assert abs(Decimal(nll) / _term(n / r, n) - 1) < Decimal(1e-13)
    for r in (1e-6, 0.01, 0.6, 1.6, 30.0, 1e5):
        rc, nll, _ = ctx.eval_grad(np.array([n / r]))
        assert rc == 0 and abs(Decimal(nll) - _term(n / r, n)) <= Decimal(4 * 2.3e-16) * Decimal(n / r + n * (1 + abs(np.log(r))))
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_sum_of_many_equal_terms(precision):
    """512 histograms of 1000 equal bins in toys enough for one block each: 2000 terms per thread.  Bound: the
    FP64 roundings of such a sum (2000 x 2^-53) and the term's own error (1e-13)."""
    torch = pytest.importorskip("torch")
    from paper_1812_05686_gb300 import gsn
    J, D, T = 1000, 512, 304
    ctx = gsn.context_from_workload(_flat(J, D), precision)
    dev = torch.device("cuda", 0)
    n = 1000.0
    counts = torch.full((T, D * J), n, dtype=torch.float64, device=dev)
    wins = torch.tensor([[0, J]], dtype=torch.int32, device=dev).repeat(T, D, 1)
    ratio = torch.linspace(0.71, 1.43, T, dtype=torch.float64, device=dev)
    rate = (n / ratio * J).reshape(T, 1)
    nll, grad = torch.empty(T, dtype=torch.float64, device=dev), torch.empty(T, 1, dtype=torch.float64, device=dev)
    torch.cuda.synchronize(dev)
    assert ctx.eval_grad_batch_dev(rate, counts, wins, nll, grad) == 0, ctx.last_error()
    torch.cuda.synchronize(dev)
    got, mu = nll.cpu().numpy(), rate.cpu().numpy()[:, 0]
    for t in range(0, T, 19):
        # the bin's content is the rate times the template's value 1 / J, rounded
        ref = _term(mu[t] * (1.0 / J), n) * J * D
        assert abs(Decimal(got[t]) / ref - 1) < Decimal(3.3e-13)
    ctx.close()
