"""Scratch memory of large FP64 batches: bounded by what the column records of a launch take (32 GiB), and
launches of fewer toys where the device has less left."""
import numpy as np
import pytest

from oracle import gsn_oracle as O
from paper_1812_05686_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GIB = 1 << 30


def _batch(torch, ctx, w, n, T):
    dev = torch.device("cuda", 0)
    J = len(w["edges"][0]) - 1
    x = torch.tensor(w["theta0"], device=dev).repeat(T, 1)
    x[:, 0] *= 1 + 0.01 * (torch.arange(T, device=dev) % 7)
    args = [x, torch.tensor(n, device=dev).repeat(T, 1), torch.tensor([[0, J]], dtype=torch.int32, device=dev).repeat(T, 1, 1),
            torch.empty(T, dtype=torch.float64, device=dev), torch.empty_like(x), torch.empty(T, dtype=torch.int32, device=dev)]
    torch.cuda.synchronize(dev)
    return args


def _check(ctx, torch, args):
    torch.cuda.synchronize()
    nll, g, st = (v.cpu().numpy() for v in args[3:])
    assert not st.any()
    T = len(nll)
    for t in (7, 8, T // 2, T - 1):     # toys of equal inputs
        r = t % 7
        assert abs(nll[t] / nll[r] - 1) < 1e-13 and np.max(np.abs(g[t] - g[r])) <= 1e-12 * np.max(np.abs(g[r]))


@pytest.mark.parametrize("left", [None, 17])
def test_scratch_of_large_batches(left):
    torch = pytest.importorskip("torch")
    from paper_1812_05686_gb300 import gsn
    w = I.single_gauss(n_bins=64, n_fine=100000, e_max=0.18)
    n = I.poisson_counts(O.expected_counts(w, w["theta0"], 0), 3)
    ctx = gsn.context_from_workload(w, gsn.GSN_FP64)
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 80 * GIB:
        pytest.skip("needs 80 GiB of free device memory")
    # 12.8 MB of column records per toy: 2680 toys fill 32 GiB, 1000 take 12 GiB
    T = 2680 if left is None else 1000
    args = _batch(torch, ctx, w, n, T)
    hold = None if left is None else torch.empty(torch.cuda.mem_get_info()[0] - left * GIB, dtype=torch.uint8, device="cuda")
    free = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        assert ctx.eval_grad_batch_dev(*args) == 0, ctx.last_error()
        _check(ctx, torch, args)
    assert free - torch.cuda.mem_get_info()[0] <= 34 * GIB
    ctx.close()
    del hold
    torch.cuda.empty_cache()
