"""Performance cases: what users of this library run, through its public entry points.

The workloads are the seeded ones of paper_1812_05686_gb300/inputs.py, at the sizes of the repository's
benchmark and tests: the single-dataset Gaussian fit (900 bins x 2000 fine points), the two-dataset
scintillator fit (1000 or 1200 bins x 20000 fine points, 16 species), its free-power generalized
gamma, the Monte Carlo template fit and the slices of a multivariate fit.

A case is a dict of plain values:
  call       point    one minimiser step: Context.eval_grad (host parameters in, NLL and gradient out)
             torch    the same step inside a torch program: the autograd function on float32 CUDA parameters
             value    NLL-only steps of a fit with numeric derivatives (Context.eval at response
                      parameters that change from call to call), then the expected counts per species
             toys     a batch of pseudo-experiments, each with its own parameters, counts and fit window
                      (Context.eval_grad_batch_dev: NLL, gradient and status of every toy)
             fit      profile-likelihood fits over the rates of a batch of toys (Context.fit_rates_batch_dev)
  work       gauss | gamma | ggamma | template | slices
  precision  fp64 (the library's default) | mixed
  bins, fine, toys   histogram bins per dataset, fine energy points, toys of the batch
"""
import math

import numpy as np
import torch

from paper_1812_05686_gb300 import gsn
from paper_1812_05686_gb300 import inputs as I

_PREC = {"fp64": gsn.GSN_FP64, "mixed": gsn.GSN_MIXED}
_BAND = 9.5        # columns further than this many sigma from a bin do not enter the reference sums
_autograd = None
_stream = None


def _program_stream():
    """The program's stream: every pass is ordered on it, and the contexts work on it too."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def listed():
    def c(name, call, work, precision, bins, fine, toys=1, **kw):
        return dict(name=name, call=call, work=work, precision=precision, bins=bins, fine=fine, toys=toys, **kw)
    return [
        # the smallest everyday call: one step of a single-dataset fit at the library's defaults
        c("point_gauss_fp64", "point", "gauss", "fp64", 900, 2000),
        # the same step in a torch optimiser loop, mixed precision: launch latency is most of it
        c("torch_gauss_mixed", "torch", "gauss", "mixed", 900, 2000),
        # one step of the two-dataset fit, the reference precision that results are checked with
        c("point_gamma_fp64", "point", "gamma", "fp64", 1000, 20000),
        # the same step in a torch program, mixed precision
        c("torch_gamma_mixed", "torch", "gamma", "mixed", 1000, 20000),
        # a fit with numeric derivatives, and the validation quantity (expected counts per species)
        c("value_gamma_fp64", "value", "gamma", "fp64", 1000, 20000),
        # the toy Monte Carlo study, the benchmark's workload: ragged windows of 600..1200 bins
        c("toys_gamma_mixed", "toys", "gamma", "mixed", 1200, 20000, 8192),
        # FP64 toys: the sample with which a mixed study is validated
        c("toys_gamma_fp64", "toys", "gamma", "fp64", 1200, 20000, 128),
        # a toy study of the single-dataset Gaussian fit at the default precision
        c("toys_gauss_fp64", "toys", "gauss", "fp64", 900, 2000, 500),
        # toys of the generalized-gamma response with a free power
        c("toys_ggamma_mixed", "toys", "ggamma", "mixed", 1200, 20000, 1024),
        # toys of a Monte Carlo template fit (no detector response)
        c("toys_template_mixed", "toys", "template", "mixed", 1000, 2, 8192),
        # discovery test: profile-likelihood fits, all rates free and >= 0, every toy in its own window
        c("fit_gamma_fp64", "fit", "gamma", "fp64", 1200, 20000, 64),
        # the large multivariate fit: 4 datasets x 64 slices, per-slice response, 32 species
        c("toys_slices_mixed", "toys", "slices", "mixed", 1000, 50000, 4, slices=64, species=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["point", "torch", "value", "toys", "toys", "toys", "fit"])
    if call == "fit":
        return dict(call=call, work="gamma", precision="fp64", bins=rng.randint(300, 1200), fine=_log_int(rng, 2000, 20000),
                    toys=_log_int(rng, 3, 64))
    if call != "toys":
        work = rng.choice(["gauss", "gamma", "gamma", "ggamma"] if call != "value" else ["gauss", "gamma", "gamma"])
        precision = "mixed" if call == "torch" else "fp64"
        fine = _log_int(rng, 500, 4000) if work == "gauss" else _log_int(rng, 2000, 20000)
        return dict(call=call, work=work, precision=precision, bins=rng.randint(250, 1100), fine=fine, toys=1)
    work = rng.choice(["gauss", "gamma", "gamma", "ggamma", "template", "slices"])
    if work == "template":
        return dict(call=call, work=work, precision=rng.choice(["mixed", "fp64"]), bins=rng.randint(200, 1000), fine=2,
                    toys=_log_int(rng, 50, 8192))
    if work == "slices":
        return dict(call=call, work=work, precision="mixed", bins=rng.randint(300, 1000), fine=_log_int(rng, 5000, 50000),
                    toys=rng.randint(1, 4), slices=rng.randint(3, 64), species=rng.randint(8, 32))
    precision = rng.choice(["mixed", "fp64"]) if work != "ggamma" else rng.choice(["mixed", "mixed", "fp64"])
    top = {("gauss", "mixed"): 8192, ("gauss", "fp64"): 500, ("gamma", "mixed"): 8192, ("gamma", "fp64"): 128,
           ("ggamma", "mixed"): 1024, ("ggamma", "fp64"): 48}[work, precision]
    fine = _log_int(rng, 500, 2000) if work == "gauss" else _log_int(rng, 2000, 20000)
    return dict(call=call, work=work, precision=precision, bins=rng.randint(250, 1200 if work != "gauss" else 900),
                fine=fine, toys=_log_int(rng, 2, top))


# ------------------------------------------------------------------ inputs ----
def _workload(case):
    b, k = case["bins"], case["fine"]
    if case["work"] == "gauss":
        return I.single_gauss(n_bins=b, n_fine=k)
    if case["work"] == "template":
        return I.template_like(n_bins=b)
    if case["work"] == "slices":
        return I.multivariate_like(n_slices=case["slices"], n_bins=b, n_fine=k, n_species=case["species"])
    w = I.borexino_like(n_bins=b, n_fine=k)
    return I.with_power(w, 1.3) if case["work"] == "ggamma" else w


def _inputs(case, seed):
    """Everything that follows from the seed: the workload, parameter points, counts, windows."""
    w = _workload(case)
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    host = np.random.Generator(np.random.PCG64(int(seed)))
    D, T = len(w["edges"]), case["toys"]
    J = len(w["edges"][0]) - 1
    # the toys are drawn from the workload's generating point; a free-power study draws them from the
    # gamma response, as the benchmark does
    base = _workload(dict(case, work="gamma")) if case["work"] == "ggamma" else w
    mu0 = _expected(base, torch.as_tensor(base["theta0"], device=dev)).reshape(-1)
    theta0 = torch.as_tensor(w["theta0"], device=dev)
    z = torch.randn(T, theta0.numel(), generator=gen, device=dev, dtype=torch.float64)
    params = torch.where(theta0 != 0, theta0 * (1 + 0.01 * z), 1e-6 * z.abs())
    counts = torch.poisson(mu0.clamp_min(0).expand(T, -1).contiguous(), generator=gen)
    if case["call"] in ("toys", "fit") and case["work"] != "slices":
        width = host.integers(J // 2, J + 1, size=T)
        lo = (host.random(T) * (J - width + 1)).astype(np.int64)
        win = np.repeat(np.stack([lo, lo + width], axis=1)[:, None, :], D, axis=1)
    else:
        win = np.tile(np.array([0, J]), (T, D, 1))
    return w, params, counts, torch.as_tensor(win.astype(np.int32), device=dev)


def prepare(case, seed):
    w, params, counts, wins = _inputs(case, seed)
    T, P = params.shape
    S = w["spectra"].shape[0]
    stream = _program_stream()
    stream.wait_stream(torch.cuda.current_stream())
    # mixed toy studies ask for results that repeat bit by bit from run to run (autotune = 0)
    kw = dict(autotune=0) if case["precision"] == "mixed" and case["call"] == "toys" else {}
    single = counts[0].cpu().numpy() if T == 1 and case["call"] != "toys" else None
    ctx = gsn.context_from_workload(w, _PREC[case["precision"]], counts=single, stream=stream.cuda_stream, **kw)
    st = dict(call=case["call"], ctx=ctx)
    if case["call"] == "point":
        st["x"] = params[0].cpu().numpy()
    elif case["call"] == "torch":
        st["x"] = params[0].float().requires_grad_(True)
    elif case["call"] == "value":
        x = params[0].cpu().numpy()
        up, dn = x.copy(), x.copy()
        up[S] *= 1 + 1e-4   # the light yield's central difference
        dn[S] *= 1 - 1e-4
        st.update(up=up, dn=dn)
    else:
        st.update(params=params, counts=counts, wins=wins)
        if case["call"] == "toys":
            f = dict(dtype=torch.float64, device=params.device)
            st.update(nll=torch.empty(T, **f), grad=torch.empty(T, P, **f),
                      status=torch.empty(T, dtype=torch.int32, device=params.device))
        else:
            free = np.zeros(P, bool)
            free[np.unique(w["slot_map"][:, :S][w["slot_map"][:, :S] >= 0])] = True
            st.update(free=free, lo=np.where(free, 0.0, -np.inf), start=params, x=torch.empty_like(params))
    return st


def run(st):
    with torch.cuda.stream(_program_stream()):
        return _run(st)


def _run(st):
    global _autograd
    ctx, call = st["ctx"], st["call"]
    if call == "point":
        rc, nll, grad = ctx.eval_grad(st["x"])
        return {"nll": nll, "grad": grad, "status": rc}
    if call == "torch":
        if _autograd is None:
            _autograd = gsn.make_autograd()
        x = st["x"]
        x.grad = None
        nll = _autograd.apply(x, ctx)
        nll.backward()
        return {"nll": nll.detach(), "grad": x.grad}
    if call == "value":
        rc0, up = ctx.eval(st["up"])
        rc1, dn = ctx.eval(st["dn"])
        return {"up": up, "dn": dn, "status": [rc0, rc1], "expected": ctx.expected(st["dn"], 0)}
    if call == "toys":
        rc = ctx.eval_grad_batch_dev(st["params"], st["counts"], st["wins"], st["nll"], st["grad"], st["status"])
        return {"nll": st["nll"], "grad": st["grad"], "status": st["status"], "rc": rc}
    st["x"].copy_(st["start"])  # the fit writes the minima over its start points
    nll, iters, status = ctx.fit_rates_batch_dev(st["x"], st["counts"], st["wins"], free=st["free"], lo=st["lo"])
    return {"params": st["x"], "nll": nll, "iters": iters, "status": status}


def work(case):
    """Bytes: inputs and results once each.  Operations: one density value per (bin, fine point) pair
    inside +-5 sigma of the point's mean (10 operations: exponent, exponential, sums), a second pass for
    the gradient, and two per (bin, species) of a template fit or a rate fit's design."""
    w = _workload(dict(case, fine=min(case["fine"], 2000)))
    D, S = len(w["edges"]), w["spectra"].shape[0]
    T, J, K, P = case["toys"], case["bins"], case["fine"], int(w["n_params"])
    nbytes = 8.0 * S * K + T * (8.0 * (2 * P + 1 + D * J) + 8.0 * D) + 16.0 * D * J
    if case["work"] == "template":
        return {"bytes": nbytes + 8.0 * D * J * S, "flops": 4.0 * T * D * J * S}
    # pairs of one response group, from the means at the generating point
    th = w["theta0"]
    E = (np.arange(K) + 0.5) * (2.0 / K)
    al, be = 1 + th[S + 1] * w["birks_s0"], th[S + 1] * w["birks_s1"]
    mu = th[S] * (E / al - be / al**2 * np.log1p(al * E / be))
    sg = np.sqrt(th[S + 2] + th[S + 3] * mu + th[S + 4] * mu * mu)
    pairs = float(np.clip(np.minimum(mu + 5 * sg, J) - np.maximum(mu - 5 * sg, 0), 0, None).sum())
    groups = case["slices"] if case["work"] == "slices" else 1
    share = 0.75 if case["call"] in ("toys", "fit") and case["work"] != "slices" else 1.0  # the windows' mean width
    per = {"point": 20.0, "torch": 20.0, "toys": 20.0, "value": 2 * (8.0 + 2 * S), "fit": 8.0 + 2 * S}[case["call"]]
    flops = T * groups * share * pairs * per
    if case["call"] == "fit":
        flops += T * 10.0 * D * J * S * S  # ten Newton steps
    return {"bytes": nbytes + (8.0 * J * S if case["call"] == "value" else 0.0), "flops": flops}


# --------------------------------------------------------- plain 64-bit reference ----
def _gl(n, dev):
    x, g = np.polynomial.legendre.leggauss(n)
    return torch.as_tensor(x, device=dev), torch.as_tensor(g, device=dev)


def _spectra(w, dev):
    """Normalised spectra, shifted ones moved up by whole fine bins."""
    s = np.array(w["spectra"], float)
    tot = s.sum(axis=1, keepdims=True)
    s = np.divide(s, tot, out=np.zeros_like(s), where=tot > 0)
    dE = w["fine_centres"][1] - w["fine_centres"][0]
    for i in np.nonzero(np.asarray(w["kind"]) == I.KIND_ANA_SHIFT)[0]:
        m = int(round(w["shift"][i] / dE))
        s[i] = np.concatenate([np.zeros(min(m, s.shape[1])), s[i][:max(s.shape[1] - m, 0)]])
    return torch.as_tensor(s, device=dev)


def _moments(w, th, q, dev):
    """Mean and variance of every fine column for the response slots q of theta."""
    E = torch.as_tensor(w["fine_centres"], device=dev)
    al, be = 1 + q[1] * w["birks_s0"], q[1] * w["birks_s1"]
    mu = q[0] * (E / al - be / al**2 * torch.log1p(al * E / be))
    return mu, q[2] + q[3] * mu + q[4] * mu * mu


def _shape(mu, var, p):
    """(d, ln s) of the generalized gamma of power p by moment matching; one Newton step carries the derivatives."""
    a = 1 / p
    t, g = _gl(24, mu.device)
    t, g = (t + 1) / 2, g / 2
    def ratio(x):   # lnGamma(x + 2a) + lnGamma(x) - 2 lnGamma(x + a) = int_0^2a psi1(x + v) min(v, 2a - v) dv, from x + 8
        v, y = a * t, x + 8
        left = (torch.special.polygamma(1, y[:, None] + v) * v) @ g
        right = (torch.special.polygamma(1, y[:, None] + 2 * a - v) * v) @ g
        return a * (left + right) - sum(torch.log1p(-(a / (x + i + a))**2) for i in range(8))
    def slope(x):
        v, y = a * t, x + 8
        low = sum(2 * a * a / ((x + i) * (x + i + a) * (x + i + 2 * a)) for i in range(8))
        return a * ((torch.special.polygamma(2, y[:, None] + v) * v) @ g +
                    (torch.special.polygamma(2, y[:, None] + 2 * a - v) * v) @ g) - low
    r = torch.log1p(var / mu**2)
    with torch.no_grad():
        x = a * a / r
        for _ in range(40):
            h = ratio(x)
            x = x * torch.exp(torch.clamp(-torch.log(h / r) * h / (x * slope(x)), -3, 3))
        sl = slope(x)
    x = x - (ratio(x) - r) / sl
    lg = a * (torch.digamma(x[:, None] + 8 + a * t) @ g) - sum(torch.log1p(a / (x + i)) for i in range(8))
    return p * x, torch.log(mu) - lg


def _response(res, mu, var, p, lo, hi):
    """Bin integrals of the response, bins [lo, hi) (edges, first bin at 0 allowed) x columns."""
    if res == I.RES_GAUSS:
        sg = torch.sqrt(var)
        z0, z1 = (lo[:, None] - mu) / sg, (hi[:, None] - mu) / sg
        up = (z0 + z1) >= 0
        a = torch.where(up, z0, -z1) / math.sqrt(2.0)
        b = torch.where(up, z1, -z0) / math.sqrt(2.0)
        return 0.5 * (torch.erfc(a) - torch.erfc(b))
    if res == I.RES_GAMMA:
        d, ls, lgd = mu * mu / var, torch.log(var / mu), None
        pw = None
    else:
        d, ls = _shape(mu, var, p)
        pw = p
    lgd = torch.lgamma(d if pw is None else d / pw)
    out = []
    zero = bool(lo[0] <= 0)
    low = int((lo < 16).sum())
    if zero:  # P(a, y) of the bin at zero by its power series
        aa = d if pw is None else d / pw
        y = torch.exp((torch.log(hi[0]) - ls) * (1 if pw is None else pw))
        term = torch.ones_like(aa)
        tot = torch.ones_like(aa)
        for n in range(1, 100):
            term = term * y / (aa + n)
            tot = tot + term
        out.append((torch.exp(aa * torch.log(y) - y - torch.lgamma(aa + 1)) * tot)[None])
    for j0, j1, n in ((int(zero), low, 20), (low, lo.numel(), 8)):
        if j1 <= j0:
            continue
        t, g = _gl(n, mu.device)
        l, h = lo[j0:j1, None], hi[j0:j1, None]
        if n == 20:   # nodes in ln x
            u = torch.log(l) + torch.log(h / l) * (t + 1) / 2
            x = torch.exp(u)
            wt = g / 2 * torch.log(h / l) * x
        else:
            x = l + (h - l) * (t + 1) / 2
            u = torch.log(x)
            wt = g / 2 * (h - l)
        acc = 0
        for i in range(n):
            ui, xi = u[:, i, None], x[:, i, None]
            if pw is None:
                e = (d - 1) * (ui - ls) - ls - xi / torch.exp(ls) - lgd
            else:
                e = torch.log(pw) - ls + (d - 1) * (ui - ls) - torch.exp(pw * (ui - ls)) - lgd
            acc = acc + wt[:, i, None] * torch.exp(e)
        out.append(acc)
    return torch.cat(out)


def _groups(w):
    """Datasets that share edges and response multipliers, with their slots."""
    S = w["spectra"].shape[0]
    scale = w.get("resp_scale")
    found = {}
    for d in range(len(w["edges"])):
        sl = [int(w["slot_map"][d, S + i]) for i in range(5)] + [int(w["slot_map"][d, 3 * S + 5])]
        key = (tuple(sl), None if scale is None else tuple(scale[d]))
        found.setdefault(key, []).append(d)
    return [(list(k[0]), k[1], ds) for k, ds in found.items()]


def _blocks(mu, var, lo, hi, size):
    """(columns, bins) blocks that hold every pair within the band."""
    sg = torch.sqrt(var).detach()
    mu, var = mu.detach(), var.detach()
    a = torch.searchsorted(hi, (mu - _BAND * sg).clamp_min(0).flip(0).cummin(0).values.flip(0).contiguous()).cpu().numpy()
    # the lowest means have a small shape and a long exponential tail of scale var / mu
    b = torch.searchsorted(lo, (mu + 1.2 * _BAND * sg + 40 * var / mu).contiguous()).cpu().numpy()
    for k0 in range(0, mu.numel(), size):
        k1 = min(mu.numel(), k0 + size)
        j0, j1 = int(a[k0:k1].min()), min(int(b[k0:k1].max()), lo.numel())
        if j1 > j0:
            yield k0, k1, j0, j1


def _slots(w, th, grp, dev):
    sl, sc, _ = grp
    q = [th[i] if i >= 0 else None for i in sl]
    if sc is not None:
        q = [v * float(sc[i]) for i, v in enumerate(q[:5])] + q[5:]
    return q


def _rates(w, th, d):
    S = w["spectra"].shape[0]
    f = torch.as_tensor(np.asarray(w["mask"])[:, d] * w["exposure"][d] * (1.0 if w.get("rate_factor") is None else w["rate_factor"][d]),
                        device=th.device, dtype=torch.float64)
    idx = torch.as_tensor(np.maximum(w["slot_map"][d, :S], 0).astype(np.int64), device=th.device)
    return f * th[idx]


def _direct(w, th, d, n):
    """Expected counts of dataset d that do not pass the response: peaks and templates, bins x species."""
    S = w["spectra"].shape[0]
    e = torch.as_tensor(np.asarray(w["edges"][d], float), device=th.device)
    out = torch.zeros(n, S, device=th.device, dtype=torch.float64)
    for s in range(S):
        if w["kind"][s] == I.KIND_ANA_PEAK and w["mask"][s, d]:
            m, wd = th[int(w["slot_map"][d, S + 5 + 2 * s])], th[int(w["slot_map"][d, S + 6 + 2 * s])]
            out = out + _response(I.RES_GAUSS, m[None], (wd * wd)[None], None, e[:-1], e[1:]) * torch.nn.functional.one_hot(
                torch.tensor(s, device=th.device), S)
        elif w["kind"][s] == I.KIND_MC_TEMPLATE and w["templates"][s] and w["templates"][s][d] is not None:
            h = torch.as_tensor(np.asarray(w["templates"][s][d], float), device=th.device)
            out[:, s] = h / h.sum()
    return out


def _smeared(w):
    return [s for s in range(w["spectra"].shape[0]) if w["kind"][s] < I.KIND_ANA_PEAK]


def _expected(w, th, per_species=None):
    """Expected counts [dataset][bin] at theta; with per_species = d, bins x species of dataset d."""
    dev = th.device
    S, D, J = w["spectra"].shape[0], len(w["edges"]), len(w["edges"][0]) - 1
    out = torch.zeros(D, J, device=dev, dtype=torch.float64)
    res = int(w["resolution"])
    with torch.no_grad():
        sp = _spectra(w, dev) if _smeared(w) else None
        shapes = None
        if sp is not None:
            for grp in _groups(w):
                if per_species is not None and per_species not in grp[2]:
                    continue
                q = _slots(w, th, grp, dev)
                e = torch.as_tensor(np.asarray(w["edges"][grp[2][0]], float), device=dev)
                mu, var = _moments(w, th, q, dev)
                T = sp[_smeared(w)].T if per_species is not None else torch.stack(
                    [(_rates(w, th, d)[_smeared(w)] @ sp[_smeared(w)]) for d in grp[2]], 1)
                acc = torch.zeros(J, T.shape[1], device=dev, dtype=torch.float64)
                for k0, k1, j0, j1 in _blocks(mu, var, e[:-1], e[1:], max(1000, mu.numel() // 8)):
                    acc[j0:j1] += _response(res, mu[k0:k1], var[k0:k1], q[5], e[j0:j1], e[j0 + 1:j1 + 1]) @ T[k0:k1]
                if per_species is not None:
                    shapes = acc
                else:
                    out[grp[2]] = acc.T
        if per_species is not None:
            d = per_species
            full = _direct(w, th, d, J)
            if shapes is not None:
                full[:, _smeared(w)] = shapes
            return full * _rates(w, th, d)
        for d in range(D):
            out[d] += _direct(w, th, d, J) @ _rates(w, th, d)
    return out


def _nll_grad(w, th0, counts, wins, grad=True):
    """NLL and gradient at one point: expected counts, then the weights 1 - n/mu pulled back block by block."""
    dev = th0.device
    D, J = len(w["edges"]), len(w["edges"][0]) - 1
    mu = _expected(w, th0)
    n = counts.reshape(-1)[:D * J].reshape(D, J)
    j = torch.arange(J, device=dev)
    inside = (j >= wins[:, :1]) & (j < wins[:, 1:])
    term = torch.where(n > 0, mu - n + n * torch.log(torch.where(n > 0, n, 1.0) / mu), mu)
    nll = torch.where(inside, term, 0.0).sum()
    th = th0.clone().requires_grad_(True)
    pulls = 0
    for i, p in enumerate(w["pull_param"]):
        pulls = pulls + 0.5 * ((th[int(p)] - float(w["pull_centre"][i])) / float(w["pull_width"][i]))**2
    value = float((nll + pulls).detach())
    if not grad:
        return value, None
    wt = torch.where(inside, 1 - n / mu, 0.0)
    res = int(w["resolution"])
    total = pulls + sum((wt[d] @ _direct(w, th, d, J)) @ _rates(w, th, d) for d in range(D))
    if _smeared(w):
        sp = _spectra(w, dev)[_smeared(w)]
        for grp in _groups(w):
            q = _slots(w, th, grp, dev)
            e = torch.as_tensor(np.asarray(w["edges"][grp[2][0]], float), device=dev)
            m, v = _moments(w, th, q, dev)
            T = torch.stack([_rates(w, th, d)[_smeared(w)] @ sp for d in grp[2]], 1)
            W = wt[grp[2]].T
            leaf = [x.detach().requires_grad_(True) for x in (m, v, T)]
            p = None if q[5] is None else q[5].detach().requires_grad_(True)
            for k0, k1, j0, j1 in _blocks(leaf[0], leaf[1], e[:-1], e[1:], max(1000, m.numel() // 8)):
                R = _response(res, leaf[0][k0:k1], leaf[1][k0:k1], p, e[j0:j1], e[j0 + 1:j1 + 1])
                ((W[j0:j1].T @ R).T * leaf[2][k0:k1]).sum().backward()
            total = total + (m * leaf[0].grad).sum() + (v * leaf[1].grad).sum() + (T * leaf[2].grad).sum()
            if p is not None:
                total = total + q[5] * p.grad
    g, = torch.autograd.grad(total, th)
    return value, g


def exact(case, seed):
    if case["call"] == "fit":     # an iterative minimum, defined by its stopping rule
        return None
    heavy = {"gauss": 0.3, "gamma": 1.0, "ggamma": 6.0, "template": 0.05, "slices": 1.0}[case["work"]]
    points = case["toys"] * case.get("slices", 1)
    if points * heavy * (0.05 + case["bins"] * case["fine"] / 2.4e7) > 150:
        return None
    w, params, counts, wins = _inputs(case, seed)
    dev = params.device
    if case["call"] == "value":
        S = w["spectra"].shape[0]
        up, dn = params[0].clone(), params[0].clone()
        up[S] *= 1 + 1e-4
        dn[S] *= 1 - 1e-4
        return {"up": _nll_grad(w, up, counts[0], wins[0], False)[0], "dn": _nll_grad(w, dn, counts[0], wins[0], False)[0],
                "status": [0, 0], "expected": _expected(w, dn, per_species=0)}
    if case["call"] == "torch":
        params = params.float().double()   # the point that the float32 parameters hold
    got = [_nll_grad(w, params[t], counts[t], wins[t]) for t in range(case["toys"])]
    if case["call"] == "toys":
        return {"nll": torch.tensor([v for v, _ in got], dtype=torch.float64, device=dev), "grad": torch.stack([g for _, g in got]),
                "status": torch.zeros(case["toys"], dtype=torch.int32, device=dev), "rc": 0}
    nll, g = got[0]
    if case["call"] == "torch":
        return {"nll": torch.tensor(nll, dtype=torch.float64), "grad": g}
    return {"nll": nll, "grad": g.cpu().numpy(), "status": 0}
