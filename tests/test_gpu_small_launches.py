"""Launches too small for the GPU split their columns over clusters and deal their column blocks to several
thread blocks; a batch large enough is evaluated without either.  Both add in the same order: the same bits."""
import numpy as np
import pytest

from paper_1812_05686_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# column blocks of 256: one, two (the second of one column), ten; dealt to as many thread blocks as there are
# column blocks (3 toys), to fewer (700 toys: four) or to one (2500 toys)
@pytest.mark.parametrize("precision", ["FP64", "MIXED"])
@pytest.mark.parametrize("J,K,power", [(40, 250, 0), (33, 257, 0), (60, 2500, 0), (60, 2500, 1.3)])
def test_small_and_large_fits_have_the_same_bits(J, K, power, precision):
    torch = pytest.importorskip("torch")
    from paper_1812_05686_gb300 import gsn
    w = I.borexino_like(n_bins=J, n_fine=K, e_max=1.2 * J / 500.0 + 0.05)
    if power:
        w = I.with_power(w, power)
    dev, T, few = torch.device("cuda", 0), 2500, 3
    ctx = gsn.context_from_workload(w, getattr(gsn, "GSN_" + precision))
    free = np.zeros(w["n_params"], bool)
    free[[w["slot_map"][0, 0], w["slot_map"][0, 1]]] = True
    mu = torch.tensor(np.concatenate([ctx.expected(w["theta0"], d).sum(axis=1) for d in range(2)]), device=dev)
    assert mu.shape == (2 * J,)
    gen = torch.Generator(device=dev)
    gen.manual_seed(5)
    counts = torch.poisson(mu.clamp_min(0).expand(T, -1).contiguous(), generator=gen)
    wins = torch.tensor([[[0, J], [0, J]]] * T, dtype=torch.int32, device=dev)
    lo = np.where(free, 0.0, -np.inf)
    out = []
    for n in (T, 700, few):
        x = torch.tensor(np.repeat(w["theta0"][None], n, axis=0), device=dev)
        nll, iters, status = ctx.fit_rates_batch_dev(x, counts[:n].contiguous(), wins[:n].contiguous(), free, lo=lo)
        torch.cuda.synchronize(dev)
        out.append([v[:few].cpu().numpy() for v in (x, nll, iters, status)])
    assert np.all(np.isfinite(out[0][1]))
    for a, b, c in zip(*out):
        assert np.array_equal(a, b) and np.array_equal(a, c)
