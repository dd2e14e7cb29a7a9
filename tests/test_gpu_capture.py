"""Steps inside a caller's CUDA graph (the work that a step runs beside the adjoint on a stream of its own
joins the capture), and the no-allocation step of a problem whose pair records do not fit its array."""
import ctypes as C

import numpy as np
import pytest

from oracle import gsn_oracle as O
from paper_1812_05686_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("peaks", [False, True])
def test_batch_in_a_callers_graph(precision, peaks):
    torch = pytest.importorskip("torch")
    from paper_1812_05686_gb300 import gsn
    w = I.borexino_like(n_bins=130, n_fine=500, e_max=0.4) if peaks else I.single_gauss(n_bins=130, n_fine=500, e_max=0.4)
    D, T, dev = len(w["edges"]), 3, torch.device("cuda", 0)
    n = np.concatenate([I.poisson_counts(O.expected_counts(w, w["theta0"], d), 3 + d) for d in range(D)])
    st = torch.cuda.Stream()
    ctx = gsn.context_from_workload(w, precision, counts=n, stream=st.cuda_stream)
    f = dict(dtype=torch.float64, device=dev)
    P = w["n_params"]
    x, counts = torch.empty(T, P, **f), torch.tensor(n, device=dev).repeat(T, 1)
    wins = torch.tensor([[0, 130]], dtype=torch.int32, device=dev).repeat(T, D, 1)
    nll, g, status = torch.empty(T, **f), torch.empty(T, P, **f), torch.empty(T, dtype=torch.int32, device=dev)
    points = [torch.tensor(I.perturbed_points(w["theta0"], T, s), device=dev) for s in (5, 6, 7)]
    x.copy_(points[0])
    torch.cuda.synchronize(dev)
    assert ctx.eval_grad_batch_dev(x, counts, wins, nll, g, status) == 0, ctx.last_error()
    torch.cuda.synchronize(dev)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        assert ctx.eval_grad_batch_dev(x, counts, wins, nll, g, status) == 0, ctx.last_error()
    for p in points:
        x.copy_(p)
        nll.fill_(np.nan), g.fill_(np.nan), status.fill_(9)
        torch.cuda.synchronize(dev)
        graph.replay()
        torch.cuda.synchronize(dev)
        got = nll.clone(), g.clone(), status.clone()
        torch.cuda.synchronize(dev)
        assert ctx.eval_grad_batch_dev(x, counts, wins, nll, g, status) == 0
        torch.cuda.synchronize(dev)
        for a, b in zip(got, (nll, g, status)):
            assert torch.equal(a, b)
    ctx.close()


def test_noalloc_without_room_for_pairs():
    """72000 columns: 11.5 MB of FP64 records fit the array of 16 MiB, 6.9 MB of pair records beside them do not."""
    torch = pytest.importorskip("torch")
    from paper_1812_05686_gb300 import gsn
    w = I.borexino_like(n_bins=60, n_fine=72000, e_max=0.2)
    w = dict(w, edges=w["edges"][:1], exposure=w["exposure"][:1], mask=w["mask"][:, :1], slot_map=w["slot_map"][:1],
             win_lo=w["win_lo"][:1], win_hi=w["win_hi"][:1])
    n = I.poisson_counts(O.expected_counts(w, w["theta0"], 0), 3)
    ctx = gsn.context_from_workload(w, gsn.GSN_FP64, counts=n)
    dev = torch.device("cuda", 0)
    for p in I.perturbed_points(w["theta0"], 2, 41):
        rc, ref, gref = ctx.eval_grad(p)
        assert rc == 0, ctx.last_error()
        x, out = torch.tensor(p, device=dev), torch.full((1 + p.size,), np.nan, dtype=torch.float64, device=dev)
        st = torch.full((1,), 9, dtype=torch.int32, device=dev)
        torch.cuda.synchronize(dev)
        ptr = lambda t, k=0: C.c_void_p(t.data_ptr() + 8 * k)
        assert ctx.lib.gsn_eval_grad_noalloc(ctx.h, ptr(x), ptr(out), ptr(out, 1), ptr(st)) == 0, ctx.last_error()
        torch.cuda.synchronize(dev)
        assert int(st) == 0 and abs(float(out[0]) - ref) <= 1e-10 * abs(ref)
        assert np.max(np.abs(out[1:].cpu().numpy() - gref)) <= 1e-8 * max(np.max(np.abs(gref)), 1.0)
    ctx.close()
