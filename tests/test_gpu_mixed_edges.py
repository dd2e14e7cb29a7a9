"""Mixed kernels at the sizes where their work is split another way: segments below the first linear bin
taken by a block, batches shared among warps (few toys of many bins), two bins per instruction of the
generalized gamma (odd windows, its two series ranges, one to four datasets), and the Poisson term's
switch between its series and the logarithm."""
import numpy as np
import pytest

from oracle import gsn_oracle as O
from paper_1812_05686_gb300 import inputs as I
from tests.test_gpu_pair64 import TWO_WIDTHS, _gamma, _gauss, _merged, _with_edges

pytestmark = pytest.mark.gpu

CASES = {
    "gauss_33": lambda: _gauss(33, 200), "gamma_64": lambda: _gamma(64, 300), "gamma_65_one_dataset": lambda: _merged(_gamma(65, 130), 1),
    "gamma_130_three": lambda: _merged(_gamma(130, 500), 3), "gamma_two_widths": lambda: _with_edges(_gamma(90, 260), TWO_WIDTHS),
    "gamma_above_zero": lambda: _with_edges(_gamma(120, 300), np.arange(20.0, 121.0)),
    "ggamma_one_dataset": lambda: I.with_power(_merged(_gamma(97, 300), 1), 1.3), "ggamma_65": lambda: I.with_power(_gamma(65, 130), 1.6),
    "ggamma_four_datasets": lambda: I.with_power(_merged(_gamma(150, 400), 4), 0.8),
    "ggamma_two_widths": lambda: I.with_power(_with_edges(_gamma(90, 260), TWO_WIDTHS), 1.2),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("toys", [3, 40])
def test_batches_against_fp64(name, toys):
    """40 toys: two bins per lane and shared batches (gamma); 3: one bin per lane.  Bounds: |dNLL| < 1e-3, and 1e-4 of
    max(|g| + sqrt(F), 1) per component, the mixed gradient's bound in windows of few bins."""
    from paper_1812_05686_gb300 import gsn
    w = CASES[name]()
    D, J = len(w["edges"]), len(w["edges"][0]) - 1
    mu = [O.expected_counts(w, w["theta0"], d) for d in range(D)]
    F = O.fisher_diagonal(w, w["theta0"])
    rng = np.random.default_rng(7)
    counts = np.stack([np.concatenate([rng.poisson(m) for m in mu]) for _ in range(toys)]).astype(float)
    params = I.perturbed_points(w["theta0"], toys, 11)
    wins = np.empty((toys, D, 2), np.int32)
    for t in range(toys):
        lo = [0, 3, J // 2, J - 33 if J > 33 else 0][t % 4]
        wins[t] = [lo, [J, J, lo + 21, J - 1][t % 4] if lo + 21 <= J else J]
    out = []
    for prec in (gsn.GSN_FP64, gsn.GSN_MIXED):
        ctx = gsn.context_from_workload(w, prec, autotune=0)
        rc, nll, g = ctx.eval_grad_batch(params, counts, wins)
        assert rc == 0, ctx.last_error()
        out.append((nll, g))
        ctx.close()
    (n64, g64), (nm, gm) = out
    assert np.max(np.abs(nm - n64)) < 1e-3
    assert np.max(np.abs(gm - g64) / np.maximum(np.abs(g64) + np.sqrt(F), 1.0)) < 1e-4


@pytest.mark.parametrize("precision", [0, 1])
def test_poisson_term_over_ratios(precision):
    """Template fit of one species, counts at ratios n / mu around the series' range (0.67 .. 1.5), at 0 and far away;
    reference in 50 digits where available (mpmath), FP64 otherwise.  Bound: 8 roundings of the largest addend."""
    from paper_1812_05686_gb300 import gsn
    ratios = [0.0, 1e-3, 0.3, 0.6, 0.66, 0.667, 0.67, 0.9, 0.999, 1.0, 1.001, 1.2, 1.49, 1.5, 1.51, 2.0, 40.0]
    for scale in (3.0, 1e3, 1e7):
        J = len(ratios)
        w = I.template_like(n_bins=J, n_species=1)
        w = dict(w, templates=[[np.ones(J)] * 2], exposure=np.ones(2))
        rate = scale * J
        n = np.rint(np.array(ratios) * scale)
        n = np.concatenate([n, n + 1])
        ctx = gsn.context_from_workload(w, precision, counts=n)
        rc, nll, g = ctx.eval_grad(np.array([rate]))
        assert rc == 0, ctx.last_error()
        m = np.longdouble(rate) / J
        x = n.astype(np.longdouble)
        ref = np.where(x > 0, m - x + x * np.log(np.where(x > 0, x, 1) / m), m).sum()
        gref = ((1 - x / m) / J).sum()
        assert abs(float(nll - ref)) <= 8 * 2.3e-16 * 40 * scale * 2 * J
        assert abs(float(g[0] - gref)) <= (1e-12 if precision == 0 else 1e-6) * float(np.abs((1 - x / m) / J).sum())
        ctx.close()
