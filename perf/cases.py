"""The solver calls that are measured, and the inputs they are measured on.

Each case is one call (or one short run of calls) that a segmentation program
makes through ``paper_2004_11227_gb300.cmf``: a solve to a certified gap, a
fixed number of iterations, a certificate evaluation, a batch solve.  Images
are the repository's synthetic recipes (disk, painted shapes, Voronoi cells,
plus noise), drawn on the GPU from the seed.  ``exact`` repeats the call in
float64 with plain torch, written from the iterations' formulas.
"""
import math

import numpy as np
import torch

from paper_2004_11227_gb300 import cmf

ALGOS = {"pADMMI": cmf.PADMM, "rpADMMI": cmf.RPADMM_FG, "rpADMMII": cmf.RPADMM_EB,
         "rPDRQ": cmf.RPDRQ, "pADMM-TY": cmf.TY, "ALG1": cmf.CP}
STORAGE = {"float32": cmf.F32, "float16": cmf.F16, "bfloat16": cmf.BF16}


def _case(name, call, model, H, W, L=2, **kw):
    d = {"name": name, "call": call, "model": model, "H": H, "W": W, "L": L,
         "recipe": "shapes" if model == "binary" else "voronoi", "algo": "rpADMMII",
         "storage": "float32", "field": True, "aniso": False, "iters": 10}
    d.update(kw)
    return d


def listed():
    return [
        # an icon-sized mask refined in an interactive loop: the solve's latency
        _case("binary_disk_64_solve", "solve", "binary", 64, 64, recipe="disk", field=False,
              iters=30),
        # the usual two-label segmentation of one camera image, edge-weighted
        _case("binary_shapes_1024_solve", "solve", "binary", 1024, 1024, iters=70),
        # a large two-label image advanced between a viewer's updates
        _case("binary_shapes_4096_iterate", "iterate", "binary", 4096, 4096, iters=20),
        # the paper's fastest two-label method on the same kind of image
        _case("binary_rpdrq_1024_iterate", "iterate", "binary", 1024, 1024, algo="rPDRQ",
              iters=20),
        # a cropped scan: odd width, ragged height, the primal-dual method
        _case("binary_odd_901x1407_iterate", "iterate", "binary", 901, 1407, algo="ALG1",
              iters=20),
        # the usual four-label segmentation, whole call
        _case("potts4_2048_solve", "solve", "potts", 2048, 2048, 4, field=False, iters=220),
        # the same labels under rPDRQ
        _case("potts4_rpdrq_2048_iterate", "iterate", "potts", 2048, 2048, 4, algo="rPDRQ",
              field=False, iters=10),
        # the many-label workload in its two flow storages (a two-phase solve
        # runs 16-bit flows first, float32 after)
        _case("potts16_4096_f32_iterate", "iterate", "potts", 4096, 4096, 16, iters=10),
        _case("potts16_4096_f16_iterate", "iterate", "potts", 4096, 4096, 16,
              storage="float16", iters=10),
        # a cropped scan with eight labels: odd width, ragged height
        _case("potts8_odd_721x1283_iterate", "iterate", "potts", 721, 1283, 8, iters=20),
        # the certificate a program asks for before it accepts a labelling
        _case("potts16_2048_certificates", "certificates", "potts", 2048, 2048, 16, iters=20),
        # a queue of images of uneven size and label count solved together
        _case("batch_12_solve", "batch", "mixed", 64, 640, 8, count=12, sizes=4,
              recipe="shapes", iters=400),
    ]


#: label-pixels x iterations of the largest listed case, the bound on drawn ones
_MOST = 4096 * 4096 * 16 * 10


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["binary_iterate", "binary_iterate", "potts_iterate", "potts_iterate",
                       "potts_iterate", "binary_solve", "potts_solve", "certificates", "batch"])
    field = rng.random() < 0.6
    aniso = rng.random() < 0.15
    algo = rng.choice(["rpADMMII"] * 4 + ["rpADMMI", "pADMMI", "pADMM-TY", "ALG1", "rPDRQ"])
    storage = rng.choice(["float32"] * 3 + ["float16"])
    if kind == "batch":
        hi = _log_int(rng, 128, 640)
        c = _case("", "batch", "mixed", 64, hi, 8, count=rng.randint(4, 12),
                  sizes=rng.randrange(1 << 20), recipe="shapes", iters=400)
    elif kind == "binary_solve":
        c = _case("", "solve", "binary", _log_int(rng, 48, 1200), _log_int(rng, 48, 1200),
                  field=field, algo=algo, aniso=aniso, iters=100)
    elif kind == "binary_iterate":
        c = _case("", "iterate", "binary", _log_int(rng, 48, 4096), _log_int(rng, 48, 4096),
                  field=field, algo=algo, aniso=aniso, storage=storage,
                  iters=rng.choice([5, 10, 20]))
    elif kind == "potts_solve":
        c = _case("", "solve", "potts", _log_int(rng, 48, 700), _log_int(rng, 48, 700),
                  rng.choice([3, 4, 8]), field=field, aniso=aniso, iters=400)
    elif kind == "certificates":
        c = _case("", "certificates", "potts", _log_int(rng, 48, 2048), _log_int(rng, 48, 2048),
                  rng.randint(2, 16), field=field, algo=algo, aniso=aniso, storage=storage,
                  iters=10)
    else:
        c = _case("", "iterate", "potts", _log_int(rng, 48, 4096), _log_int(rng, 48, 4096),
                  rng.choice([2, 3, 4, 4, 6, 8, 11, 16, 16, 24]), field=field, algo=algo,
                  aniso=aniso, storage=storage, iters=rng.choice([5, 10, 20]))
    if c["model"] == "potts" and c["L"] == 2 and c["algo"] == "ALG1":
        c["algo"] = "rpADMMII"  # its default step is the two-label model's
    while c["call"] == "iterate" and c["H"] * c["W"] * c["L"] * c["iters"] > _MOST:
        c["H"] = c["H"] * 7 // 10
    del c["name"]
    return c


# --- inputs ------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _levels(L):
    if L == 4:
        return [0.1, 0.4, 0.6, 0.9]
    return [i / (L - 1) for i in range(L)]


def _image(case, L, H, W, seed):
    """The noisy image (float64, on the GPU) and its label levels."""
    g = np.random.RandomState(seed % (1 << 31))
    ii = torch.arange(H, device="cuda", dtype=torch.float64)[:, None]
    jj = torch.arange(W, device="cuda", dtype=torch.float64)[None, :]
    if case["recipe"] == "disk":
        levels, sigma = [0.2, 0.8], 0.1
        rad = 20.0 * min(H, W) / 64.0
        ci, cj = (H - 1) / 2 + g.uniform(-2, 2), (W - 1) / 2 + g.uniform(-2, 2)
        img = torch.where((ii - ci) ** 2 + (jj - cj) ** 2 <= rad * rad, 0.8, 0.2).double()
    elif case["recipe"] == "shapes":
        sigma = 0.15
        levels = [0.2, 0.8] if L == 2 else [0.1 + 0.8 * i / (L - 1) for i in range(L)]
        img = torch.full((H, W), levels[0], device="cuda", dtype=torch.float64)
        for _ in range(8):
            ci, cj = g.uniform(0, H), g.uniform(0, W)
            r = g.uniform(32.0, 160.0) * min(H, W) / 1024.0
            if g.rand() < 0.5:
                m = (ii - ci) ** 2 + (jj - cj) ** 2 <= r * r
            else:
                m = ((ii - ci).abs() <= r) & ((jj - cj).abs() <= r)
            img = torch.where(m, levels[g.randint(1, L)], img)
    else:
        levels, sigma = _levels(L), 0.1 if L <= 8 else 0.05
        n = max(8, round(64 * H * W / 2048 ** 2))
        best = torch.full((H, W), 1e30, device="cuda")
        img = torch.zeros((H, W), device="cuda", dtype=torch.float64)
        for _ in range(n):
            ci, cj, lev = g.uniform(0, H), g.uniform(0, W), levels[g.randint(0, L)]
            d = (ii - ci).float() ** 2 + (jj - cj).float() ** 2
            img = torch.where(d < best, lev, img)
            best = torch.minimum(best, d)
    noise = torch.randn((H, W), device="cuda", dtype=torch.float64, generator=_gen(seed))
    return img + sigma * noise, levels


def _instance(case, model, L, H, W, seed):
    """(costs float32 [2 or L, H, W], alpha float or float32 [H, W]), on the GPU."""
    img, levels = _image(case, L, H, W, seed)
    if model == "binary":
        costs = torch.stack([(img - 0.2).abs(), (img - 0.8).abs()]).float()
        base = 0.5
    else:
        costs = torch.stack([((img - c) ** 2).float() for c in levels])
        base = 0.5 if case["recipe"] == "shapes" else 0.3
    if not case["field"]:
        return costs, base
    dx = torch.zeros_like(img)
    dy = torch.zeros_like(img)
    dx[:, :-1] = img[:, 1:] - img[:, :-1]
    dy[:-1] = img[1:] - img[:-1]
    return costs, (base * torch.exp(-10.0 * torch.sqrt(dx * dx + dy * dy))).float()


def _batch_shapes(case, seed):
    """(model, L, H, W, seed) of each image; the sizes belong to the case."""
    g = np.random.RandomState(case["sizes"])
    out = []
    for k in range(case["count"]):
        side = int(g.randint(case["H"], case["W"] + 1))
        L = [2, 3, 4, case["L"]][k % 4]
        out.append(("binary" if L == 2 else "potts", L, side, side, seed + 7919 * (k + 1)))
    return out


def _problem(case, model, L, H, W, seed, params):
    costs, alpha = _instance(case, model, L, H, W, seed)
    costs = costs.cpu().numpy()
    alpha = alpha if isinstance(alpha, float) else alpha.cpu().numpy()
    if model == "binary":
        return cmf.Binary(costs[0], costs[1], alpha, params)
    return cmf.Potts(costs, alpha, params)


def _params(case, L):
    kw = {"storage": STORAGE[case["storage"]], "aniso": int(case["aniso"])}
    if case["call"] in ("solve", "batch"):
        kw.update(tol_gap=1e-4, max_iter=2000, check_every=20 if case["call"] == "batch" else 10)
    return cmf.default_params(ALGOS[case["algo"]], L, **kw)


def prepare(case, seed):
    if case["call"] == "batch":
        p = _params(case, 2)
        items = [_problem(case, *s, p) for s in _batch_shapes(case, seed)]
        return {"case": case, "items": items, "batch": cmf.Batch(items, p)}
    p = _params(case, case["L"])
    s = _problem(case, case["model"], case["L"], case["H"], case["W"], seed, p)
    if case["call"] != "solve":
        (cmf.cmf_init_binary if case["model"] == "binary" else cmf.cmf_init_potts)(s)
    if case["call"] == "certificates":
        cmf.cmf_iterate_potts(s, case["iters"])
    return {"case": case, "problem": s}


def _state(s):
    names = ("u", "qx", "qy", "ps", "pt") if isinstance(s, cmf.Binary) else \
        ("u", "qx", "qy", "p", "ps")
    return {k: getattr(s, k) for k in names}


def run(state):
    case = state["case"]
    if case["call"] == "batch":
        status, res = state["batch"].solve()
        return {"states": [_state(s) for s in state["items"]], "status": status,
                "iterations": np.array([r["iters"] for r in res]),
                "energy": np.array([r["energy"] for r in res], dtype=np.float32)}
    s = state["problem"]
    binary = case["model"] == "binary"
    if case["call"] == "certificates":
        return cmf.cmf_eval_potts(s)
    if case["call"] == "iterate":
        (cmf.cmf_iterate_binary if binary else cmf.cmf_iterate_potts)(s, case["iters"])
        return _state(s)
    status, iters, hist = (cmf.cmf_solve_binary if binary else cmf.cmf_solve_potts)(s)
    return {"state": _state(s), "status": status, "iterations": iters,
            "energy": float(hist[-1, 1]), "dual": float(hist[-1, 2])}


def work(case):
    """Costs and alpha read once, the state written once (and, unless the call
    starts cold, read once); arithmetic of the iterations' formulas, counted
    per label and pixel (per pixel for the two-label model)."""
    es = 4 if case["storage"] == "float32" else 2
    shapes = _batch_shapes(case, 1) if case["call"] == "batch" else \
        [(case["model"], case["L"], case["H"], case["W"], 0)]
    nbytes = flops = 0.0
    for model, L, H, W, _ in shapes:
        n = H * W
        if model == "binary":
            inputs, state, per_it, per_check = 8 * n, (4 + 4 * es) * n, 52 * n, 50 * n
        else:
            inputs, state = 4 * L * n, (L * (4 + 3 * es) + 4) * n
            per_it, per_check = (46 * L + 4) * n, (40 + 2 * L) * L * n
        if case["algo"] == "rPDRQ":
            per_it *= 1.2
        inputs += 4 * n if case["field"] else 0
        if case["call"] == "certificates":
            nbytes += inputs + state + 32
            flops += per_check
        elif case["call"] == "iterate":
            nbytes += inputs + 2 * state
            flops += per_it * case["iters"]
        else:  # "iters" is then about what a solve to the gap takes
            nbytes += inputs + state
            flops += (per_it + per_check / 10) * case["iters"]
    return {"bytes": float(nbytes), "flops": float(flops)}


# --- the same calls in float64 -----------------------------------------------------

def _grad(v):
    gx, gy = torch.zeros_like(v), torch.zeros_like(v)
    gx[..., :-1] = v[..., 1:] - v[..., :-1]
    gy[..., :-1, :] = v[..., 1:, :] - v[..., :-1, :]
    return gx, gy


def _div(qx, qy):
    d = torch.zeros_like(qx)
    d[..., :-1] += qx[..., :-1]
    d[..., 1:] -= qx[..., :-1]
    d[..., :-1, :] += qy[..., :-1, :]
    d[..., 1:, :] -= qy[..., :-1, :]
    return d


def _project(x, y, alpha, aniso):
    if aniso:
        return torch.clamp(x, -alpha, alpha), torch.clamp(y, -alpha, alpha)
    n = torch.sqrt(x * x + y * y)
    s = torch.where(n > alpha, alpha / torch.clamp(n, min=1e-300), torch.ones_like(n))
    return x * s, y * s


class _Exact:
    """One problem in float64: the cold start, the iterations, the certificates."""

    def __init__(self, case, model, L, H, W, seed):
        costs, alpha = _instance(case, model, L, H, W, seed)
        self.C = costs.double()
        self.alpha = torch.full((H, W), np.float32(alpha).item(), device="cuda",
                                dtype=torch.float64) if isinstance(alpha, float) else alpha.double()
        self.binary, self.L, self.algo = model == "binary", L, case["algo"]
        self.aniso, self.pitch, self.W = case["aniso"], cmf.pitch_for(W), W
        self.p = p = _params(case, 2 if case["call"] == "batch" else L)
        self.sigma, self.tau = p.sigma, p.tau
        self.a2 = max(p.a2, 2.0 * L)
        i = torch.arange(H, device="cuda")[:, None] + torch.arange(W, device="cuda")[None, :]
        self.red = i % 2 == 0
        n = torch.full((H, W), 4.0, device="cuda", dtype=torch.float64)
        n[0] -= 1
        n[-1] -= 1
        n[:, 0] -= 1
        n[:, -1] -= 1
        self.nb = n
        self._cold()

    def _cold(self):
        dr = self.algo == "rPDRQ"
        if self.binary:
            cs, ct = self.C
            u, m = (ct < cs).double(), torch.minimum(cs, ct)
            self.ps, self.pt = m.clone(), m.clone()
        else:
            m, best = self.C.min(0)
            first = (self.C == m).double().argmax(0) if self.L > 1 else best
            u = torch.zeros_like(self.C).scatter_(0, first[None], 1.0)
            self.ps, self.p_ = m.clone(), m.expand_as(self.C).clone()
        self.u, self.qx, self.qy = u, torch.zeros_like(u), torch.zeros_like(u)
        if dr:
            gx, gy = _grad(u)
            self.qx, self.qy = self.tau * gx, self.tau * gy
            if self.binary:
                self.pt, self.ps = self.pt - self.tau * u, self.ps + self.tau * u
            else:
                self.p_, self.ps = self.p_ - self.tau * u, self.ps + self.tau

    def _sweep(self, b, u, kappa):
        st = self.sigma * self.tau
        for red in (True, False, True):
            s = torch.zeros_like(u)
            s[..., 1:] += u[..., :-1]
            s[..., :-1] += u[..., 1:]
            s[..., 1:, :] += u[..., :-1, :]
            s[..., :-1, :] += u[..., 1:, :]
            v = (b / st + s) / (kappa + self.nb)
            u = torch.where(self.red if red else ~self.red, v, u)
        return u

    def _flows(self, u):
        gx, gy = _grad(u)
        x, y = self.qx - self.tau * gx, self.qy - self.tau * gy
        tx, ty = _project(2 * x - self.qx, 2 * y - self.qy, self.alpha, self.aniso)
        self.qx = self.qx + self.p.rho * (tx - x)
        self.qy = self.qy + self.p.rho * (ty - y)

    def _step_dr(self):
        p, tau = self.p, self.tau
        d = _div(self.qx, self.qy)
        if self.binary:
            u = self._sweep(-self.sigma * (d + self.pt - self.ps), self.u, 2.0)
        else:
            st = self.sigma * tau
            b = -self.sigma * (d + self.p_ - self.ps) + st * (self.L * self.u - self.u.sum(0))
            u = self._sweep(b, self.u, self.L + 1.0)
        self._flows(u)
        if self.binary:
            t, s = self.pt + tau * u, self.ps - tau * u
            self.pt = self.pt + p.rho * (torch.minimum(2 * t - self.pt, self.C[1]) - t)
            self.ps = self.ps + p.rho * (torch.minimum(2 * s - self.ps + tau, self.C[0]) - s)
        else:
            t, s = self.p_ + tau * u, self.ps - tau * u.sum(0)
            self.p_ = self.p_ + p.rho * (torch.minimum(2 * t - self.p_, self.C) - t)
            self.ps = self.ps + p.rho * (2 * s - self.ps + tau - s)
        self.u = u

    def _step(self):
        if self.algo == "rPDRQ":
            return self._step_dr()
        p, al = self.p, self.algo
        rho = p.rho if al == "rpADMMII" else 1.0
        omr = 1.0 - p.rho if al == "rpADMMII" else 0.0
        cu = p.r * p.c if al == "rpADMMI" else p.c
        ic = 1.0 / (self.tau if al == "ALG1" else p.c)
        step = self.sigma * self.tau if al == "ALG1" else 1.0 / p.a
        pt, ps, u = (self.pt if self.binary else self.p_), self.ps, self.u
        g = _div(self.qx, self.qy) + pt - ps - u * ic
        gx, gy = _grad(g)
        self.qx, self.qy = _project(self.qx + step * gx, self.qy + step * gy, self.alpha,
                                    self.aniso)
        d = _div(self.qx, self.qy)
        del gx, gy
        cap = self.C[1] if self.binary else self.C
        if al == "ALG1":
            ub = -self.tau * g
            pt1 = torch.minimum(pt + self.sigma * ub, cap)
            if self.binary:
                ps1 = torch.minimum(ps - self.sigma * ub + self.sigma, self.C[0])
            else:
                ps1 = ps - self.sigma * ub.sum(0) + self.sigma
            u1 = u - self.tau * (d + pt1 - ps1)
        elif al == "pADMM-TY":
            if self.binary:
                ps1 = torch.minimum(pt + d - u * ic + ic, self.C[0])
                pt1 = torch.minimum(ps1 - d + u * ic, cap)
            else:
                pt1 = torch.minimum(ps - d + u * ic, cap)
                ps1 = ((pt1 + d - u * ic).sum(0) + ic) / self.L
            u1 = u - cu * (pt1 - ps1 + d)
        else:
            r = rho * (pt - ps) - u * ic + rho * d
            pt1 = torch.minimum(pt - r / p.a1, cap)
            if self.binary:
                ps1 = torch.minimum(ps + (r + ic) / p.a1, self.C[0])
            else:
                ps1 = ps + (r.sum(0) + ic) / self.a2
            u1 = u - cu * ((pt1 - ps1) - omr * (pt - ps) + rho * d)
        self.u, self.ps = u1, ps1
        if self.binary:
            self.pt = pt1
        else:
            self.p_ = pt1

    def iterate(self, n):
        for _ in range(n):
            self._step()
        return self

    def certificates(self):
        u, x, y = self.u, self.qx, self.qy
        pt, ps = (self.pt if self.binary else self.p_), self.ps
        if self.algo == "rPDRQ":
            gx, gy = _grad(u)
            x, y = x - self.tau * gx, y - self.tau * gy
            pt, ps = pt + self.tau * u, ps - self.tau * (u if self.binary else u.sum(0))
        res = (_div(x, y) - ps + pt).square().sum().sqrt()
        px, py = _project(x, y, self.alpha, self.aniso)
        if self.binary:
            ub = u.clamp(0, 1)
            E = ((1 - ub) * self.C[0] + ub * self.C[1]).sum()
            D = torch.minimum(self.C[0], self.C[1] + _div(px, py)).sum()
        else:
            s, _ = u.sort(0, descending=True)
            k = torch.arange(1, self.L + 1, device="cuda", dtype=torch.float64)[:, None, None]
            t = (s.cumsum(0) - 1) / k
            n = (s > t).sum(0, keepdim=True)
            ub = (u - t.gather(0, n - 1)).clamp(min=0)
            E = (ub * self.C).sum()
            D = (self.C + _div(px, py)).min(0)[0].sum()
        gx, gy = _grad(ub)
        tv = gx.abs() + gy.abs() if self.aniso else torch.sqrt(gx * gx + gy * gy)
        E = float(E + (self.alpha * tv).sum())
        D = float(D)
        return E, D, (E - D) / max(abs(E), 1e-30), float(res)

    def solve(self):
        it, p = 0, self.p
        while it < p.max_iter:
            self.iterate(p.check_every)
            it += p.check_every
            E, D, gap, _ = self.certificates()
            if gap <= p.tol_gap:
                break
        return E, D

    def state(self):
        names = {"u": self.u, "qx": self.qx, "qy": self.qy, "ps": self.ps}
        names["pt" if self.binary else "p"] = self.pt if self.binary else self.p_
        return {k: torch.nn.functional.pad(v, (0, self.pitch - self.W))
                for k, v in names.items()}


def exact(case, seed):
    if case["call"] == "batch":
        if sum(L * H * W for _, L, H, W, _ in _batch_shapes(case, seed)) > 4_000_000:
            return None  # hundreds of float64 iterations of every instance: over 20 seconds
        ex = [_Exact(case, *s) for s in _batch_shapes(case, seed)]
        energy = np.array([x.solve()[0] for x in ex])
        return {"states": [x.state() for x in ex], "status": None, "iterations": None,
                "energy": energy}
    x = _Exact(case, case["model"], case["L"], case["H"], case["W"], seed)
    if case["call"] == "solve":
        E, D = x.solve()
        return {"state": x.state(), "status": None, "iterations": None, "energy": E, "dual": D}
    x.iterate(case["iters"])
    return x.certificates() if case["call"] == "certificates" else x.state()
