"""The FP64 response in pairs against the plain FP64 kernels, at bounds near the pairs' own error.  A
secondary observable whose shapes are all zero contributes nothing and selects the plain FP64 kernels.
Bounds: a pair's density is good to a few 2^-48 of its exponent's terms (tens), 1e-13; ten times that on
expected counts, per species and relative wherever a bin holds more than 1e-6 of the species' largest; on
the NLL, whose sum of |mu - n| grows with the bins; five times that again on gradient components, against
their own value and the square root of the Fisher information.  A gamma-family column's derivatives are what
remains of terms that cancel at its moments: 2e2 times as large for the mean (LY, kB), 2e3 times for the
variance (a, b, c) and 1e4 times and more for the free power, here; 1e-13 times that there."""
import numpy as np
import pytest

from oracle import gsn_oracle as O
from paper_1812_05686_gb300 import inputs as I
from tests.test_gpu_pair64 import TWO_WIDTHS, _merged, _with_edges

pytestmark = pytest.mark.gpu

CASES = {
    "gauss": lambda: I.single_gauss(n_bins=300, n_fine=900, e_max=0.75),
    "gauss_wide": lambda: _with_edges(I.single_gauss(n_bins=300, n_fine=900, e_max=0.75), np.arange(0.0, 300.5, 0.5)),
    "gamma": lambda: I.borexino_like(n_bins=300, n_fine=2500, e_max=0.75),
    "gamma_three": lambda: _merged(I.borexino_like(n_bins=200, n_fine=900, e_max=0.5), 3),
    "gamma_two_widths": lambda: _with_edges(I.borexino_like(n_bins=90, n_fine=500, e_max=0.25), TWO_WIDTHS),
    "ggamma": lambda: I.with_power(I.borexino_like(n_bins=200, n_fine=900, e_max=0.5), 1.3),
    "ggamma_low_power": lambda: I.with_power(I.borexino_like(n_bins=200, n_fine=900, e_max=0.5), 0.8),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_pairs_against_plain_fp64(name):
    from paper_1812_05686_gb300 import gsn
    w = CASES[name]()
    D, S, J = len(w["edges"]), w["spectra"].shape[0], len(w["edges"][0]) - 1
    mu = [O.expected_counts(w, w["theta0"], d) for d in range(D)]
    n = np.concatenate([I.poisson_counts(m, 31 + d) for d, m in enumerate(mu)])
    F = O.fisher_diagonal(w, w["theta0"])
    points = I.perturbed_points(w["theta0"], 3, 77)
    wins = np.array([[[0, J]] * D, [[J // 3, J - 5]] * D, [[0, J // 2]] * D], np.int32)
    out = []
    for plain in (True, False):
        ctx = gsn.context_from_workload(w, gsn.GSN_FP64, counts=n)
        if plain:
            ctx.set_secondary(0, [0, 1], np.zeros((S, 1, 1)))
        rc, nll, g = ctx.eval_grad_batch(points, np.tile(np.append(n, [0.0] * plain), (3, 1)), wins)
        assert rc == 0, ctx.last_error()
        out.append((nll, g, [ctx.expected(points[0], d) for d in (0, D - 1)]))
        ctx.close()
    (n64, g64, e64), (nll, g, e) = out
    assert np.max(np.abs(nll / n64 - 1)) < 1e-12
    tol = np.full(g.shape[1], 5e-12)
    if int(w["resolution"]) != I.RES_GAUSS:
        slots = w["slot_map"][0]
        tol[slots[S:S + 2]] = 2e-11
        tol[slots[S + 2:S + 5]] = 2e-10
        if int(w["resolution"]) == I.RES_GGAMMA:
            tol[slots[3 * S + 5]] = 1e-9
    assert np.all(np.abs(g - g64) <= tol * (np.abs(g64) + np.sqrt(F)))
    for a, b in zip(e, e64):
        top = b.max(axis=0)
        assert np.all(np.abs(a - b) <= 1e-12 * top)
        big = b > 1e-6 * top
        assert np.all(np.abs(a - b)[big] <= 1e-12 * b[big])
