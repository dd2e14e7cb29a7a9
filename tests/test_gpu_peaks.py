"""AnaPeak species anywhere in the species list (a warp finds them, 32 species at a time), with profiles
inside the histogram, cut by either end, narrower than a bin and outside; FP64 path against the oracle
with its tolerances (1e-10 relative on the NLL, 1e-8 normwise on the gradient)."""
import numpy as np
import pytest

from oracle import gsn_oracle as O
from paper_1812_05686_gb300 import inputs as I
from tests._helpers import norm_rel

pytestmark = pytest.mark.gpu

PROFILES = [(60.0, 7.0), (2.0, 5.0), (118.5, 4.0), (40.3, 0.2), (31.0, 3.0), (90.0, 11.0), (400.0, 3.0), (75.0, 2.0)]


@pytest.mark.parametrize("S,peaks", [(9, (8,)), (9, (0, 3)), (32, (0, 31)), (33, (31, 32)), (64, (0, 1, 30, 31, 32, 33, 62, 63))])
def test_peaks_against_oracle(S, peaks):
    from paper_1812_05686_gb300 import gsn
    J = 120
    w = I.single_gauss(n_bins=J, n_fine=160, e_max=0.33)
    kind = np.zeros(S, np.int32)
    kind[list(peaks)] = 2
    prof = PROFILES[:len(peaks)]
    theta0 = np.concatenate([np.full(S, 40.0) + 3.0 * np.arange(S), w["theta0"][8:13], np.ravel(prof)])
    w.update(spectra=w["spectra"][np.arange(S) % 8], kind=kind, shift=np.zeros(S), mask=np.ones((S, 1), np.uint8),
             n_params=theta0.size, slot_map=I._slot_map_shared(S, 1, peaks=peaks), theta0=theta0,
             param_names=[f"r{s}" for s in range(S)] + ["LY", "kB", "a", "b", "c"] + [f"q{i}" for i in range(2 * len(peaks))])
    n = I.poisson_counts(O.expected_counts(w, theta0, 0), 3)
    p = I.perturbed_points(theta0, 1, 5)[0]
    ctx = gsn.context_from_workload(w, gsn.GSN_FP64, counts=n)
    rc, nll, g = ctx.eval_grad(p)
    assert rc == 0, ctx.last_error()
    ref, gref = O.nll(w, p, n), O.nll_grad(w, p, n)
    assert abs(nll - ref) <= 1e-10 * max(abs(ref), 1.0)
    assert norm_rel(g, gref) < 1e-8
    wins = np.array([[[5, 61]], [[58, 120]]], np.int32)
    rc, nl, gr = ctx.eval_grad_batch(np.tile(p, (2, 1)), np.tile(n, (2, 1)), wins)
    for t in range(2):
        ref, gref = O.nll(w, p, n, wins[t]), O.nll_grad(w, p, n, wins[t])
        assert abs(nl[t] - ref) <= 1e-10 * max(abs(ref), 1.0)
        assert norm_rel(gr[t], gref) < 1e-8
    ctx.close()
