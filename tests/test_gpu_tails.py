"""Counts far outside the spectrum, in bins whose tile of 32 a column's band still reaches: the expectation
there lies far below FP32's range (10 to 20 sigma beyond the last column), and the FP64 precision evaluates
it with the FP64 formulas.  Reference: the oracle, which has no band, with the FP64 path's tolerances (1e-10
relative on the NLL, 1e-8 on the gradient, here relative to every component's own value or 1).  The oracle's
gradient of a gamma response differentiates the distribution function, which is 1 to all digits out there: for
the bins beyond the spectrum it is taken from central differences of its log expectations (1e-12 of scipy's
incomplete gamma over steps of 1e-3), and the tolerance is 1e-7 (five nodes per bin in tails that fall
by e^3 per bin: 2e-8)."""
import ctypes as C

import numpy as np
import pytest

from oracle import gsn_oracle as O
from paper_1812_05686_gb300 import inputs as I
from tests.test_gpu_pair64 import _merged

pytestmark = pytest.mark.gpu


def _work(e_max, a, b, resolution=I.RES_GAUSS, power=None, datasets=1):
    w = I.single_gauss(n_bins=128, n_fine=300, e_max=e_max)
    th = w["theta0"].copy()
    th[8 + 2], th[8 + 3] = a, b
    w = dict(w, theta0=th, resolution=resolution)
    if power:
        w = I.with_power(w, power)
    return _merged(w, datasets) if datasets > 1 else w


# workload, bins with one count beyond the spectrum, and the bin with 200
CASES = {
    # sigma of 3 bins, last column at 55.4: 9.7 to 12.5 sigma (quadrature in pairs)
    "gauss": (lambda: _work(0.12, 9.0, 0.0), [84, 86, 88], 92),
    # sigma of 1.6 bins, last column at 61.3: 15 to 19 sigma; 200 counts there over an expectation below 1e-80
    "gauss_narrow": (lambda: _work(0.132, 2.6, 0.0), [86, 88], 91),
    # sigma of 6.5 bins, last column at 56: smooth columns, 9.6 to 10.7 sigma (columns that do not reach the
    # tile, which the oracle has, are 1e-10 of the expectation there)
    "gauss_smooth": (lambda: _work(0.1213, 42.0, 0.0), [118, 121], 125),
    "gauss_two_datasets": (lambda: _work(0.12, 9.0, 0.0, datasets=2), [85], 91),
    "gauss_four_datasets": (lambda: _work(0.12, 9.0, 0.0, datasets=4), [85], 91),
    "gamma": (lambda: _work(0.094, 0.001, 0.25, I.RES_GAMMA), [84, 88], 94),
    "ggamma": (lambda: _work(0.094, 0.001, 0.3, I.RES_GAMMA, power=1.2), [84], 92),
}


def _data(w, stray, many):
    n = [I.poisson_counts(O.expected_counts(w, w["theta0"], d), 5 + d) for d in range(len(w["edges"]))]
    for d, x in enumerate(n):
        assert np.all(x[min(stray):] == 0)
        if d == len(n) - 1:      # the other datasets of the group hold nothing there
            x[stray] = 1
            x[many] = 200
    # window up to the last count: the oracle's expectations further out underflow
    w["win_hi"] = np.full(len(n), many + 1, np.int32)
    return many + 1, np.concatenate(n)


def _grad(w, p, n, wins=None):
    """Gradient: the oracle's, bins from 64 on of gamma responses by differences of the expectations."""
    if int(w["resolution"]) == I.RES_GAUSS:
        return O.nll_grad(w, p, n, wins)
    lo, hi = (int(w["win_lo"][0]), int(w["win_hi"][0])) if wins is None else (int(wins[0][0]), int(wins[0][1]))
    g = O.nll_grad(w, p, n, [[lo, max(lo, min(hi, 64))]])
    j = np.arange(max(lo, 64), max(hi, 64))
    mu = O.expected_counts(w, p, 0)[j]
    for i in range(p.size):
        h = {w["spectra"].shape[0] + 2: 4e-4, w["spectra"].shape[0] + 4: 1e-6}.get(i, 1e-3 * abs(p[i]))   # a = 1e-3, c = 0
        def f(k):
            q = p.copy()
            q[i] += k * h
            return np.log(O.expected_counts(w, q, 0)[j] / mu)
        g[i] += np.sum((mu - n[j]) * (8 * (f(1) - f(-1)) - (f(2) - f(-2))) / (12 * h))
    return g


def _close(w, nll, g, ref, gref):
    assert np.isfinite(nll) and np.all(np.isfinite(g))
    assert abs(nll - ref) <= 1e-10 * abs(ref)
    assert np.max(np.abs(g - gref) / np.maximum(np.abs(gref), 1.0)) < (1e-8 if int(w["resolution"]) == I.RES_GAUSS else 1e-7)


@pytest.mark.parametrize("name", sorted(CASES))
def test_counts_outside_the_spectrum(name):
    from paper_1812_05686_gb300 import gsn
    torch = pytest.importorskip("torch")
    make, stray, many = CASES[name]
    w = make()
    J, n = _data(w, stray, many)
    D, th = len(w["edges"]), w["theta0"]
    ref, gref = O.nll(w, th, n), _grad(w, th, n)
    ctx = gsn.context_from_workload(w, gsn.GSN_FP64, counts=n)
    rc, nll, g = ctx.eval_grad(th)
    assert rc == 0, ctx.last_error()
    _close(w, nll, g, ref, gref)
    # the value alone: from new shapes, from cached ones, and after another point has used the scratch
    for _ in range(2):
        rc, v = ctx.eval(th)
        assert rc == 0 and abs(v - ref) <= 1e-10 * abs(ref), ctx.last_error()
    other = th.copy()
    other[8] *= 1.02
    ctx.eval_grad(other)
    rates = th.copy()
    rates[:8] *= 1.1
    rc, v = ctx.eval(rates)
    assert rc == 0 and abs(v - O.nll(w, rates, n)) <= 1e-10 * abs(ref)
    # expected counts: no more than the response gives, however small that is
    e, eref = ctx.expected(th, D - 1), O.expected_per_species(w, th, D - 1)
    assert np.all(np.abs(e - eref) <= 1e-10 * np.max(eref))
    far = eref < 1e-30 * np.max(eref)
    assert np.any(far) and np.all(e[far] <= 1.05 * eref[far])
    # batches: every count in the window, some, none; windows that cut the tile or start with it
    last = max(stray + [many])
    wins = np.array([[[0, J]] * D, [[7, last]] * D, [[3, min(stray)]] * D, [[min(stray) // 32 * 32, last + 1]] * D], np.int32)
    P = I.perturbed_points(th, 4, 91, 0.001)
    rc, nl, gr = ctx.eval_grad_batch(P, np.tile(n, (4, 1)), wins)
    assert rc == 0, ctx.last_error()
    for t in range(4):
        _close(w, nl[t], gr[t], O.nll(w, P[t], n, wins[t]), _grad(w, P[t], n, wins[t]))
    # without allocation
    dev = torch.device("cuda", 0)
    x = torch.tensor(th, device=dev)
    out = torch.zeros(1 + th.size, dtype=torch.float64, device=dev)
    st = torch.full((1,), 9, dtype=torch.int32, device=dev)
    torch.cuda.synchronize(dev)
    ptr = lambda t, k=0: C.c_void_p(t.data_ptr() + 8 * k)
    assert ctx.lib.gsn_eval_grad_noalloc(ctx.h, ptr(x), ptr(out), ptr(out, 1), ptr(st)) == 0, ctx.last_error()
    torch.cuda.synchronize(dev)
    assert int(st) == 0
    _close(w, float(out[0]), out[1:].cpu().numpy(), ref, gref)
    ctx.close()
