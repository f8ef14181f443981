"""Measured cases: the calls that a program makes into this library, at the sizes it makes them.

A case names one entry point (``op``) with its sizes, network, precision and options.  ``prepare``
draws the data on the GPU from the seed, ``run`` makes the call, and ``exact`` solves the same
problem in 64 bits with plain torch (a working-set solver with a closed-form last step, sharing no
code with the library).

Networks are those of the library's own workloads: AR(1) with 0.4, Erdos-Renyi with edge
probability 3/p and magnitudes in [0.1, 0.4], hubs with weight 0.25 (scaled to the fit: at most
p/10 hubs of p/4 links), AR(4) with 0.6^d, and AR(1) with 0.48 (the estimation study's chain).
"""
import math

import numpy as np
import torch

import paper_2203_15031_gb300 as sp

DEV = "cuda"
BATCH_KINDS = ("ar1", "er", "hub")


def listed():
    return [
        # The smallest fit a program makes: one double-precision estimate on a chain graph.
        # Launches, latency of one column's chain, the call itself.
        dict(name="fit_ar1_p100_fp64", op="fit", net="ar1", p=100, n=50, prec="fp64", tol=1e-8,
             center=False, diag=False),
        # An ordinary single estimate in single precision (Gram on the CUDA cores, then the fit).
        dict(name="fit_er_p2000_fp32", op="fit", net="er", p=2000, n=200, prec="fp32", tol=1e-6,
             center=False, diag=False),
        # A centred estimate at an odd size whose result is checked on the device, as a caller of
        # the mixed mode reads the error stated with its result.
        dict(name="fit_hub_p1003_mixed_diag", op="fit", net="hub", p=1003, n=251, prec="mixed",
             tol=1e-6, center=True, diag=True),
        # The largest single estimate: hub network, heavy columns, tensor-core Gram.
        dict(name="fit_hub_p10000_mixed", op="fit", net="hub", p=10000, n=500, prec="mixed",
             tol=1e-6, center=False, diag=False),
        # The headline batch: 256 fits of mixed sizes in one captured graph.
        dict(name="batch256_mixed", op="batch", count=256, p_lo=50, p_hi=2000, n_lo=30, n_hi=400,
             shapes=1000, net="mix", prec="mixed", tol=1e-6, graph=True, rule="univ"),
        # A batch of equal, larger fits.
        dict(name="batch_er_p2000_x10_mixed", op="batch", count=10, p_lo=2000, p_hi=2000, n_lo=200,
             n_hi=200, shapes=0, net="er", prec="mixed", tol=1e-6, graph=True, rule="univ"),
        # One cell of an estimation study: many double-precision fits of one network and size.
        dict(name="study_ar4_p500_x50_fp64", op="batch", count=50, p_lo=500, p_hi=500, n_lo=250,
             n_hi=250, shapes=0, net="ar4", prec="fp64", tol=1e-8, graph=False, rule="ub"),
        # One scaled-lasso regression: a single column's chain behind a Gram.
        dict(name="lasso_p2000_mixed", op="lasso", net="er", p=2000, n=200, prec="mixed", tol=1e-6),
        # The fit without a Gram matrix, for data whose p x p matrices are not wanted.
        dict(name="residual_er_p2000_fp32", op="residual", net="er", p=2000, n=200, prec="fp32",
             tol=1e-6),
        # The Gram alone at the study's largest size, on the CUDA cores.
        dict(name="gram_p5000_n1000_fp32", op="gram", net="ar1", p=5000, n=1000, prec="fp32",
             center=False),
        # Host data in, host results out, in one call.
        dict(name="solve_er_p1500_mixed_host", op="solve", net="er", p=1500, n=300, prec="mixed",
             tol=1e-6),
        # Requests of mixed sizes served by the continuously batching context.
        dict(name="serve_x24_mixed", op="serve", count=24, p_lo=100, p_hi=5000, shapes=7, net="mix",
             prec="mixed", tol=1e-6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["fit", "fit", "fit", "batch", "batch", "study", "lasso", "residual", "gram",
                     "solve", "serve"])
    net = rng.choice(["ar1", "er", "hub"])
    if op == "fit":
        prec = rng.choice(["fp32", "mixed", "mixed", "fp64"])
        p = _log_int(rng, 50, 600 if prec == "fp64" else 9000)
        return dict(op="fit", net=net, p=p, n=_log_int(rng, 40, 500), prec=prec,
                    tol=1e-8 if prec == "fp64" else 1e-6, center=rng.random() < 0.3,
                    diag=prec == "mixed" and rng.random() < 0.3)
    if op == "batch":
        p_hi = _log_int(rng, 200, 2000)
        return dict(op="batch", count=_log_int(rng, 4, 200), p_lo=max(20, p_hi // rng.randint(2, 30)),
                    p_hi=p_hi, n_lo=30, n_hi=rng.randint(60, 400), shapes=rng.randrange(1 << 20),
                    net="mix", prec=rng.choice(["mixed", "mixed", "fp32"]), tol=1e-6,
                    graph=rng.random() < 0.7, rule="univ")
    if op == "study":
        p, n = rng.randint(100, 500), rng.randint(100, 250)
        return dict(op="batch", count=rng.randint(8, 50), p_lo=p, p_hi=p, n_lo=n, n_hi=n, shapes=0,
                    net=rng.choice(["ar1_study", "ar4"]), prec="fp64", tol=1e-8, graph=False,
                    rule="ub")
    if op == "gram":
        prec = rng.choice(["fp32", "mixed", "fp64"])
        return dict(op="gram", net="ar1", p=_log_int(rng, 50, {"fp32": 5000, "mixed": 10000,
                                                               "fp64": 1500}[prec]),
                    n=_log_int(rng, 30, 1000), prec=prec, center=rng.random() < 0.3)
    if op == "serve":
        return dict(op="serve", count=rng.randint(4, 24), p_lo=100, p_hi=_log_int(rng, 300, 5000),
                    shapes=rng.randrange(1 << 20), net="mix", prec="mixed", tol=1e-6)
    if op == "lasso":
        p, n = _log_int(rng, 100, 5000), _log_int(rng, 50, 500)
    elif op == "residual":
        p, n = _log_int(rng, 50, 2000), _log_int(rng, 40, 200)
    else:
        p, n = _log_int(rng, 50, 1500), _log_int(rng, 40, 400)
    return dict(op=op, net=net, p=p, n=n, prec="fp32" if op == "residual" else "mixed", tol=1e-6)


# ----------------------------------------------------------------------------- inputs
def _shapes(c):
    """(network, p, n) of every fit of a batch or of every request, from the case alone."""
    r = np.random.default_rng(c["shapes"])
    out = []
    for i in range(c["count"]):
        p = int(round(math.exp(r.uniform(math.log(c["p_lo"]), math.log(c["p_hi"])))))
        n = int(r.integers(c["n_lo"], c["n_hi"] + 1)) if c["op"] == "batch" else max(p // 4, 50)
        kind = BATCH_KINDS[int(r.integers(0, 3))]
        out.append((kind if c["net"] == "mix" else c["net"], p, n))
    return out


def _dtype(c):
    return torch.float64 if c["prec"] == "fp64" else torch.float32


def _min_eig(E):
    """The smallest eigenvalue of a symmetric matrix, by 64 Lanczos steps."""
    p = E.shape[0]
    v = torch.cos(torch.arange(p, device=E.device, dtype=E.dtype) ** 2)
    v, old = v / v.norm(), torch.zeros_like(v)
    al, be = [], []
    for _ in range(min(64, p)):
        w = E @ v
        al.append(torch.dot(v, w))
        w = w - al[-1] * v - (be[-1] * old if be else 0.0)
        be.append(w.norm().clamp(min=1e-20))
        v, old = w / be[-1], v
    al, be = torch.stack(al), torch.stack(be)[:-1]
    t = torch.diag(al) + torch.diag(be, 1) + torch.diag(be, -1)
    return float(torch.linalg.eigvalsh(t.double().cpu())[0])


def _theta(net, p, g, dtype):
    T = torch.zeros((p, p), dtype=dtype, device=DEV)
    if net in ("ar1", "ar1_study", "ar4"):
        T.fill_diagonal_(1.0)
        for d in range(1, 5 if net == "ar4" else 2):
            v = {"ar1": 0.4, "ar1_study": 0.48, "ar4": 0.6 ** d}[net]
            T.diagonal(d).fill_(v)
            T.diagonal(-d).fill_(v)
        return T
    if net == "er":
        u = torch.rand((p, p), generator=g, device=DEV, dtype=dtype)
        m = 0.1 + 0.3 * torch.rand((p, p), generator=g, device=DEV, dtype=dtype)
        s = torch.where(torch.rand((p, p), generator=g, device=DEV) < 0.5, -1.0, 1.0).to(dtype)
        T = torch.triu(torch.where(u < 3.0 / p, m * s, torch.zeros_like(m)), 1)
        T = T + T.T
    else:
        hubs, links = min(20, max(1, p // 10)), min(50, max(1, p // 4))
        order = torch.randperm(p, generator=g, device=DEV)
        hub, rest = order[:hubs], order[hubs:]
        pick = torch.rand((hubs, rest.numel()), generator=g, device=DEV).topk(links, dim=1).indices
        T[hub[:, None], rest[pick]] = 0.25
        T = torch.maximum(T, T.T)
    shift = max(0.0, 0.1 - (1.0 + _min_eig(T)))
    return T / (1.0 + shift) + torch.eye(p, dtype=dtype, device=DEV)


def _data(net, p, n, g, dtype, sets=1):
    """sets x n rows with covariance Theta^-1: x = L^-T z for Theta = L L'."""
    L = torch.linalg.cholesky_ex(_theta(net, p, g, dtype))[0]
    Z = torch.randn((p, sets * n), generator=g, device=DEV, dtype=dtype)
    X = torch.linalg.solve_triangular(L.T, Z, upper=True).T.contiguous()
    return X if sets == 1 else list(X.reshape(sets, n, p).unbind(0))


def _lambda(c, n, p):
    return math.sqrt((4.0 if c.get("rule") == "ub" else 2.0) * math.log(p) / n)


def _inputs(c, seed):
    """The data of every fit of the case, in order."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    dt = _dtype(c)
    if c["op"] in ("batch", "serve"):
        shapes = _shapes(c)
        if len(set(shapes)) == 1 and c["prec"] == "fp64":       # one network, many datasets
            net, p, n = shapes[0]
            xs = _data(net, p, n, g, dt, len(shapes))
            return [x.contiguous() for x in xs] if isinstance(xs, list) else [xs]
        return [_data(net, p, n, g, dt) for net, p, n in shapes]
    X = _data(c["net"], c["p"], c["n"], g, dt)
    if c["op"] != "lasso":
        return [X]
    # ten coefficients of +-1 and noise 0.5
    beta = torch.zeros(c["p"], device=DEV, dtype=torch.float64)
    k = min(10, c["p"])
    at = torch.randperm(c["p"], generator=g, device=DEV)[:k]
    beta[at] = torch.where(torch.rand(k, generator=g, device=DEV) < 0.5, -1.0, 1.0).double()
    noise = torch.randn(c["n"], generator=g, device=DEV, dtype=torch.float64)
    return [X, (X.double() @ beta + 0.5 * noise).to(dt)]


def prepare(case, seed):
    c = dict(case)
    xs = _inputs(c, seed)
    s = {"c": c, "x": xs}
    if c["op"] == "batch":
        s["batch"] = sp.Batch([(x, _lambda(c, *x.shape)) for x in xs], kind="X", precision=c["prec"],
                              tol=c["tol"], maxit=1000, use_graph=c["graph"])
        # the gaps between the fits' blocks are never written
        s["batch"].Theta_buf.zero_()
        s["batch"].sigma_buf.zero_()
    elif c["op"] == "serve":
        s["server"] = sp.Server(120 << 30, max_slots=256, precision=c["prec"], tol=c["tol"],
                                maxit=1000)
        s["lam"] = [_lambda(c, *x.shape) for x in xs]
    elif c["op"] == "solve":
        s["host"] = xs[0].cpu().numpy()
    torch.cuda.synchronize()
    return s


def run(s):
    c, xs = s["c"], s["x"]
    op = c["op"]
    if op == "batch":
        s["batch"].run()
        return {"Theta": s["batch"].Theta_buf, "sigma": s["batch"].sigma_buf}
    if op == "serve":
        srv = s["server"]
        live = {srv.submit(x, lam): i for i, (x, lam) in enumerate(zip(xs, s["lam"]))}
        out = [None] * len(xs)
        while live:
            for t in list(live):
                r = srv.poll(t)
                if r is not None:
                    out[live.pop(t)] = r
        return {"Theta": [r[1] for r in out], "sigma": [r[2] for r in out]}
    n, p = xs[0].shape
    if op == "gram":
        return {"S": sp.gram(xs[0], precision=c["prec"], center=c["center"])}
    lam = _lambda(c, n, p)
    if op == "fit":
        S = sp.gram(xs[0], precision=c["prec"], center=c["center"])
        Theta, sigma, st = sp.fit(S, lam, tol=c["tol"], maxit=1000, precision=c["prec"], n=n,
                                  diagnostics=c["diag"])
        out = {"Theta": Theta, "sigma": sigma}
        if c["diag"]:
            out["err_est"] = st["err_est"]
        return out
    if op == "residual":
        Theta, sigma, _ = sp.fit_residual(xs[0], lam, tol=c["tol"], maxit=1000, precision=c["prec"])
        return {"Theta": Theta, "sigma": sigma}
    if op == "lasso":
        beta, sigma, _ = sp.scaled_lasso(xs[0], xs[1], lam, tol=c["tol"], maxit=1000,
                                         precision=c["prec"])
        return {"beta": beta, "sigma": sigma}
    Theta, sigma, _ = sp.solve(s["host"], lam, tol=c["tol"], maxit=1000, precision=c["prec"])
    return {"Theta": Theta, "sigma": sigma}


def work(case):
    """Data read once and results written once; the flops of the Gram's upper triangle (the
    coordinate descent's own depend on the data; the residual form has no Gram)."""
    c = case
    size = 8 if c["prec"] == "fp64" else 4
    shapes = _shapes(c) if c["op"] in ("batch", "serve") else [(None, c["p"], c["n"])]
    b = f = 0
    for _, p, n in shapes:
        b += size * n * p
        if c["op"] == "gram":
            b += size * p * p
        elif c["op"] == "lasso":
            b += size * n + 8 * (p + 1)
        else:
            b += 8 * p * p + 8 * p
        if c["op"] != "residual":
            f += n * p * (p + 1)
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------- 64 bits
class _Columns:
    """Scaled lassos of columns `cols` of a working matrix, each on its own candidate coordinates:
    Q (C, m, m), c (C, m), the coordinates (-1: none) and the response's own variance."""

    def __init__(self, SC, cols, lam, cand):
        C, m = cand.shape
        at = cand.clamp(min=0)
        ok = cand >= 0
        self.Q = SC[at[:, :, None], at[:, None, :]] * (ok[:, :, None] & ok[:, None, :])
        self.Q += torch.diag_embed((~ok).double())
        self.c = SC[cols[:, None], at] * ok
        self.s = SC[cols, cols]
        self.lam = torch.full((C,), float(lam), dtype=torch.float64, device=DEV)


def _polish(Q, c, s, lam, b):
    """The minimiser with the support and signs of b held, its sigma in closed form, and whether
    it satisfies every optimality condition on the candidates."""
    on = b != 0
    sg = torch.sign(b)
    M = Q * (on[:, :, None] & on[:, None, :]) + torch.diag_embed((~on).double())
    u = torch.linalg.solve(M, torch.stack([c * on, sg], dim=2))
    den = 1.0 - lam ** 2 * (sg * u[:, :, 1]).sum(1)
    var = (s - (c * u[:, :, 0] * on).sum(1)) / den
    sigma = var.clamp(min=0).sqrt()
    x = u[:, :, 0] - (lam * sigma)[:, None] * u[:, :, 1]
    x = x * on
    g = c - torch.einsum("ckm,cm->ck", Q, x)
    limit = (lam * sigma)[:, None] * (1 + 1e-9)
    good = (den > 0) & (var > 0) & (torch.sign(x) == sg).all(1) & ((g.abs() <= limit) | on).all(1)
    return x, sigma, good


def _solve_columns(Q, c, s, lam):
    C, m = c.shape
    dq = torch.diagonal(Q, dim1=1, dim2=2)
    b = torch.zeros_like(c)
    sigma = s.sqrt()
    done = torch.zeros(C, dtype=torch.bool, device=DEV)
    todo = torch.arange(C, device=DEV)
    for sweeps in (20, 40, 100, 300, 1000):
        q, cc, d, x, sig = Q[todo], c[todo], dq[todo].clone(), b[todo], sigma[todo]
        l0, ss = lam[todo], s[todo]
        g = cc - torch.einsum("ckm,cm->ck", q, x)
        for _ in range(sweeps):
            la = l0 * sig
            for k in range(m):
                t = g[:, k] + d[:, k] * x[:, k]
                nb = torch.sign(t) * (t.abs() - la).clamp(min=0) / d[:, k]
                g.addcmul_(q[:, k, :], (nb - x[:, k])[:, None], value=-1.0)
                x[:, k] = nb
            sig = (ss - (x * (cc + g)).sum(1)).clamp(min=1e-300).sqrt()
        px, ps, good = _polish(q, cc, ss, l0, x)
        b[todo] = torch.where(good[:, None], px, x)
        sigma[todo] = torch.where(good, ps, sig)
        done[todo] = good
        todo = todo[~good]
        if todo.numel() == 0:
            break
    return b, sigma, bool(done.all())


def _exact_fits(problems, m=64):
    """(B, sigma) on the working scale of every (SC, lambda0, columns), or None: candidates grow by
    the coordinates that violate the optimality conditions until there are none."""
    jobs, out = [], []
    for f, (SC, lam, cols) in enumerate(problems):
        p = SC.shape[0]
        A = SC[cols].abs()
        A[torch.arange(cols.numel(), device=DEV), cols] = -1.0
        k = min(m, p - 1)
        cand = torch.full((cols.numel(), m), -1, dtype=torch.long, device=DEV)
        cand[:, :k] = A.topk(k, dim=1).indices
        jobs.append([f, cols, cand])
        out.append([torch.zeros((cols.numel(), p), dtype=torch.float64, device=DEV),
                    torch.zeros(cols.numel(), dtype=torch.float64, device=DEV),
                    torch.arange(cols.numel(), device=DEV)])
    rows = [o[2] for o in out]
    for _ in range(12):
        parts = [_Columns(problems[f][0], cols, problems[f][1], cand) for f, cols, cand in jobs]
        b, sigma, ok = _solve_columns(*(torch.cat([getattr(x, a) for x in parts])
                                        for a in ("Q", "c", "s", "lam")))
        del parts
        if not ok:
            return None
        nxt, at = [], 0
        for f, cols, cand in jobs:
            SC, lam, _ = problems[f]
            C, p = cols.numel(), SC.shape[0]
            bf, sf = b[at:at + C], sigma[at:at + C]
            at += C
            full = torch.zeros((C, p), dtype=torch.float64, device=DEV)
            full.scatter_add_(1, cand.clamp(min=0), bf * (cand >= 0))
            out[f][0][rows[f]] = full
            out[f][1][rows[f]] = sf
            g = SC[cols] - torch.sparse.mm(full.to_sparse(), SC)
            over = g.abs() - (lam * sf)[:, None] * (1 + 1e-9)
            over.scatter_(1, cols[:, None], -1.0)
            over[full != 0] = -1.0
            bad = (over > 0).any(1)
            if bool(bad.any()):
                # violators take the places of candidates at zero
                k = min(m, p)
                v, w = over[bad].topk(k, dim=1)
                w = torch.where(v > 0, w, torch.full_like(w, -1))
                keep = torch.where(bf[bad] != 0, cand[bad], torch.full_like(cand[bad], -1))
                both = torch.cat([keep, w], dim=1)
                both = both.gather(1, (both < 0).to(torch.int8).argsort(dim=1, stable=True))
                if bool((both[:, m:] >= 0).any()):
                    return None
                rows[f] = rows[f][bad]
                nxt.append([f, cols[bad], both[:, :m].contiguous()])
        jobs = nxt
        if not jobs:
            return [(o[0], o[1]) for o in out]
    return None


def _working(X, center):
    X = X.double()
    if center:
        X = X - X.mean(0, keepdim=True)
    S = X.T @ X / X.shape[0]
    cs = S.diagonal().rsqrt()
    return S, S * cs[:, None] * cs[None, :], cs


def _assemble(B, sigma, cs):
    """Theta from B (row j: coefficients of regression j): Omega_1[:, j] = -b_j / sigma_j^2, the
    entry of smaller magnitude of each pair, back on the data's scale."""
    W = -B / (sigma ** 2)[:, None]                      # W[j, k]: entry (k, j) of Omega_1
    T = torch.where(W.abs() <= W.T.abs(), W, W.T)
    T.fill_diagonal_(0.0)
    T = T + torch.diag(sigma ** -2)
    return T * cs[:, None] * cs[None, :], sigma / cs


def exact(case, seed):
    c = dict(case)
    xs = _inputs(c, seed)
    if c["op"] == "gram":
        return {"S": _working(xs[0], c["center"])[0]}
    if c["op"] == "lasso":
        n, p = xs[0].shape
        _, SC, cs = _working(torch.cat([xs[0], xs[1][:, None]], dim=1), False)
        r = _exact_fits([(SC, _lambda(c, n, p), torch.tensor([p], device=DEV))])
        if r is None:
            return None
        B, sigma = r[0]
        return {"beta": (B[0] * cs / cs[p])[:p], "sigma": float(sigma[0] / cs[p])}
    work_ = [_working(x, c.get("center", False)) for x in xs]
    r = _exact_fits([(SC, _lambda(c, *x.shape), torch.arange(SC.shape[0], device=DEV))
                     for x, (_, SC, _) in zip(xs, work_)])
    if r is None:
        return None
    got = [_assemble(B, sigma, cs) for (B, sigma), (_, _, cs) in zip(r, work_)]
    if c["op"] == "batch":                              # the outputs' blocks start 256 bytes apart
        def packed(ts):
            size = [-(-t.numel() // 32) * 32 for t in ts]
            buf = torch.zeros(sum(size), dtype=torch.float64, device=DEV)
            at = 0
            for t, k in zip(ts, size):
                buf[at:at + t.numel()] = t.reshape(-1)
                at += k
            return buf
        return {"Theta": packed([t for t, _ in got]), "sigma": packed([s for _, s in got])}
    if c["op"] == "serve":
        return {"Theta": [t for t, _ in got], "sigma": [s for _, s in got]}
    out = {"Theta": got[0][0], "sigma": got[0][1]}
    if c["op"] == "solve":
        out = {k: v.cpu().numpy() for k, v in out.items()}
    if c.get("diag"):
        out["err_est"] = None
    return out
