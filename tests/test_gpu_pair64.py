"""FP64 path evaluated in FP32 pairs (csrc/gsn_pair64.cu) at the sizes where its rules change: tile and
batch remainders, histograms too short or too uneven for the bin-centre rule, columns too narrow for the
pairs, lines (evaluated in FP64), one to four datasets per response group, more than 16 species.  The
reference is the FP64 oracle, with the FP64 path's tolerances (1e-10 relative on the NLL, 1e-8 normwise
on the gradient, 1e-10 of the largest expected count per species)."""
import numpy as np
import pytest

from oracle import gsn_oracle as O
from paper_1812_05686_gb300 import inputs as I
from tests._helpers import norm_rel

pytestmark = pytest.mark.gpu


def _gauss(J, K, **theta):
    w = I.single_gauss(n_bins=J, n_fine=K, e_max=1.2 * J / 500.0 + 0.05)
    w["theta0"] = w["theta0"].copy()
    for k, v in theta.items():
        w["theta0"][w["param_names"].index(k)] = v
    return w


def _with_edges(w, edges):
    J = len(edges) - 1
    D = len(w["edges"])
    return dict(w, edges=[np.asarray(edges, float)] * D, win_lo=np.zeros(D, np.int32), win_hi=np.full(D, J, np.int32))


def _merged(w, n):
    """n datasets of the same response group: the first dataset repeated with other exposures."""
    rep = lambda v: np.repeat(np.asarray(v)[:1], n, axis=0)
    return dict(w, edges=[w["edges"][0]] * n, exposure=1.0 / (1.0 + np.arange(n)), mask=np.repeat(w["mask"][:, :1], n, axis=1),
                slot_map=rep(w["slot_map"]), win_lo=rep(w["win_lo"]), win_hi=rep(w["win_hi"]))


def _gamma(J, K):
    return I.borexino_like(n_bins=J, n_fine=K, e_max=1.2 * J / 500.0 + 0.05)


UNEVEN = np.concatenate([np.arange(0.0, 40.0, 2.0), 40.0 + 1.5 * np.arange(21), [75.0, 90.0]])
TWO_WIDTHS = np.concatenate([np.arange(0.0, 40.0), 40.0 + 1.25 * np.arange(41)])
CASES = {
    # bins below, at and above the shortest histogram of the bin-centre rule (16 + 32 bins), tile remainders
    "gauss_47": lambda: _gauss(47, 300), "gauss_48": lambda: _gauss(48, 300), "gauss_65": lambda: _gauss(65, 97),
    "gauss_one_batch": lambda: _gauss(128, 32), "gauss_batch_plus_one": lambda: _gauss(96, 33),
    "gauss_uneven": lambda: _with_edges(_gauss(90, 200), UNEVEN),
    # sigma below the pairs' range: FP64 formulas; around their boundary
    "gauss_narrow": lambda: _gauss(70, 200, a=0.3, b=0.01), "gauss_boundary": lambda: _gauss(70, 200, a=2.2, b=0.05),
    "gauss_fractional_bins": lambda: _with_edges(_gauss(90, 200), np.linspace(3.0, 80.0, 101)),
    "gamma_100": lambda: _gamma(100, 400), "gamma_63": lambda: _gamma(63, 129),
    "gamma_two_widths": lambda: _with_edges(_gamma(90, 200), TWO_WIDTHS),
    "gamma_above_zero": lambda: _with_edges(_gamma(120, 300), np.arange(20.0, 121.0)),
    "gamma_three_datasets": lambda: _merged(_gamma(70, 200), 3), "gamma_four_datasets": lambda: _merged(_gamma(70, 200), 4),
    "gamma_one_dataset": lambda: _merged(_gamma(70, 200), 1),
    "gamma_many_species": lambda: I.multivariate_like(n_datasets=2, n_slices=2, n_bins=80, n_fine=250, n_species=19, e_max=0.25),
    "ggamma_low_power": lambda: I.with_power(_gamma(64, 200), 0.8),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_pairs_against_oracle(name):
    from paper_1812_05686_gb300 import gsn
    w = CASES[name]()
    D, J = len(w["edges"]), len(w["edges"][0]) - 1
    mu = [O.expected_counts(w, w["theta0"], d) for d in range(D)]
    n = np.concatenate([I.poisson_counts(m, 31 + d) for d, m in enumerate(mu)])
    p = I.perturbed_points(w["theta0"], 1, 77)[0]
    ctx = gsn.context_from_workload(w, gsn.GSN_FP64, counts=n)
    rc, nll, g = ctx.eval_grad(p)
    assert rc == 0, ctx.last_error()
    ref, gref = O.nll(w, p, n), O.nll_grad(w, p, n)
    assert abs(nll - ref) <= 1e-10 * max(abs(ref), 1.0)
    assert norm_rel(g, gref) < 1e-8
    # per-species shapes, and the NLL from them
    for d in (0, D - 1):
        e = ctx.expected(p, d)
        eref = O.expected_per_species(w, p, d)
        assert np.max(np.abs(e - eref)) <= 1e-10 * max(np.max(np.abs(eref)), 1.0)
    rc, v = ctx.eval(p)
    assert rc == 0 and abs(v - ref) <= 1e-10 * max(abs(ref), 1.0)
    # windows that cut tiles and the bin-centre rule's halo
    wins = np.array([[[J // 3, J - 5]] * D, [[0, min(J, 17)]] * D, [[min(J - 1, 33), min(J, 34)]] * D], np.int32)
    P = I.perturbed_points(w["theta0"], 3, 91)
    rc, nl, gr = ctx.eval_grad_batch(P, np.tile(n, (3, 1)), wins)
    assert rc == 0, ctx.last_error()
    for t in range(3):
        ref, gref = O.nll(w, P[t], n, wins[t]), O.nll_grad(w, P[t], n, wins[t])
        assert abs(nl[t] - ref) <= 1e-10 * max(abs(ref), 1.0)
        assert norm_rel(gr[t], gref) < 1e-8
    ctx.close()
