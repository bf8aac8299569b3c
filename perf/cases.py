"""The work that users of this framework have it do, as cases that can be timed and compared.

A solve case runs a set number of PDHG iterations (tolerance out of reach, certificates tested at
every check as in a solve to tolerance), so that a pass is the same work whatever the rounding.
The adaptive step-size rule amplifies a rounding-level difference about tenfold every 40 steps, so
only the short float64 solves use it; the others keep the step size at 0.9 (||K~||_2 <= 1 after the
Pock-Chambolle scaling), and the kernels they run are the same.  Points of solves with float32
iterates are given in the iterates' precision.
"""
import math
import random

import numpy as np
import torch

import lpgen
import paper_2503_10344_gb300 as P

DEV = "cuda"


# ---------------------------------------------------------------- the cases
def _solve(name, family, m, precision, api, iters, adaptive=False, persistent=0, start="cold"):
    c = {"kind": "solve", "family": family, "m": m, "precision": precision, "api": api,
         "iters": iters, "adaptive": adaptive, "persistent": persistent, "start": start}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one MIP's relaxation from host arrays in float64: the smallest call of the heuristic
        _solve("relaxation_host_fp64", "relaxation", 200, "fp64", "host", 384),
        # the same size in the one-block form, as code that solves many small relaxations asks for
        _solve("relaxation_one_block_fp32", "relaxation", 200, "fp32", "device", 256, persistent=2),
        # a mid-sized MIP with an integer matrix, stored in bfloat16
        _solve("relaxation_mid_bf16", "relaxation", 2000, "bf16", "device", 256),
        # a small covering LP from host arrays on the 0/1 pattern: a sub-problem of the search
        _solve("cover_2k_host_pattern", "cover", 2000, "bf16", "host", 384),
        # the benchmark's covering LP
        _solve("cover_50k_pattern", "cover", 50_000, "bf16", "device", 640),
        # the same in plain float64 with default options, the comparison baseline and parity mode
        _solve("cover_50k_fp64", "cover", 50_000, "fp64", "device", 64, adaptive=True),
        # a month of the energy-system model
        _solve("energy_720h_fp32", "energy", 720, "fp32", "device", 1024),
        # the year: the largest LP the repository solves, beyond L2
        _solve("energy_8760h_fp32", "energy", 8760, "fp32", "device", 1024),
        # the uneven covering sub-LPs that partial fixings leave, solved together
        {"name": "batch_96_pattern", "kind": "batch", "count": 96, "mmin": 2000, "mmax": 40_000,
         "precision": "bf16", "iters": 128},
        # the learned start's network: one prediction
        {"name": "gnn_forward_25k", "kind": "forward", "m": 25_000},
        # a training step's gradients over a batch of four labelled graphs
        {"name": "gnn_gradient_4x12k", "kind": "gradient", "m": 12_500, "graphs": 4},
        # a solve from the learned start, from the host LP to the point
        _solve("cover_10k_learned_start", "cover", 10_000, "bf16", "host", 256, start="learned"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["relaxation", "relaxation", "cover", "cover", "cover", "energy", "energy",
                       "batch", "forward", "gradient", "learned"])
    if kind == "relaxation":
        prec = rng.choice(["fp64", "fp32", "bf16"])
        m = _log(rng, 40, 3000)
        adaptive = prec == "fp64" and rng.random() < 0.5
        return _solve("", kind, m, prec, rng.choice(["host", "device"]),
                      rng.randint(48, 64) if adaptive else rng.randint(96, 384), adaptive,
                      persistent=2 if m < 400 and rng.random() < 0.5 else 0)
    if kind == "cover":
        prec = rng.choice(["fp64", "fp32", "bf16", "bf16"])
        adaptive = prec == "fp64" and rng.random() < 0.5
        return _solve("", kind, _log(rng, 300, 60_000), prec, rng.choice(["host", "device"]),
                      rng.randint(48, 64) if adaptive else rng.randint(128, 640), adaptive)
    if kind == "energy":
        prec = rng.choice(["fp64", "fp32", "fp32"])
        adaptive = prec == "fp64" and rng.random() < 0.5
        return _solve("", kind, _log(rng, 24, 8000 if prec == "fp32" else 2000), prec,
                      rng.choice(["host", "device"]),
                      rng.randint(48, 64) if adaptive else rng.randint(128, 1024), adaptive)
    if kind == "batch":
        mmin = _log(rng, 200, 4000)
        return {"kind": "batch", "count": _log(rng, 2, 96), "mmin": mmin,
                "mmax": mmin + _log(rng, 100, 36_000), "iters": rng.randint(64, 128),
                "precision": rng.choice(["fp32", "bf16"])}
    if kind == "forward":
        return {"kind": "forward", "m": _log(rng, 200, 40_000)}
    if kind == "gradient":
        return {"kind": "gradient", "m": _log(rng, 200, 16_000), "graphs": rng.randint(1, 4)}
    return _solve("", "cover", _log(rng, 400, 30_000), "bf16", "host", rng.randint(128, 256),
                  start="learned")


# ---------------------------------------------------------------- inputs
def _cover(seed, m, fixed=False):
    """A covering LP as lpgen.set_cover and set_cover_fixed describe it (each of 4m columns covers
    3..10 rows, costs 1..100; fixed: 10-50 % of the columns fixed to 0 or 1), the pattern drawn
    and sorted on the GPU."""
    n = 4 * m
    g = torch.Generator(device=DEV).manual_seed(seed)
    k = torch.randint(3, 11, (n, 1), generator=g, device=DEV)
    rows = torch.randint(0, m, (n, 10), generator=g, device=DEV)
    take = torch.arange(10, device=DEV)[None, :] < k
    cols = torch.arange(n, device=DEV)[:, None].expand(n, 10)
    rows, cols = rows[take], cols[take]
    fill = torch.randint(0, n, (m,), generator=g, device=DEV)  # every row keeps a column
    key = torch.unique(torch.cat([rows * n + cols, torch.arange(m, device=DEV) * n + fill]))
    rows, cols = key // n, key % n
    l, u = torch.zeros(n, device=DEV), torch.ones(n, device=DEV)
    if fixed:
        frac = 0.1 + 0.4 * float(torch.rand(1, generator=g, device=DEV))
        fix = torch.rand(n, generator=g, device=DEV) < frac
        fix[fill] = False
        one = torch.rand(n, generator=g, device=DEV) < 0.5
        l[fix & one] = 1.0
        u[fix & ~one] = 0.0
    c = torch.randint(1, 101, (n,), generator=g, device=DEV).double()
    ptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    host = lambda t: t.cpu().numpy()
    return lpgen.LP(m, n, host(ptr), host(cols.int()), np.ones(cols.numel()), np.ones(m),
                    np.full(m, lpgen.SENSE_GE, dtype=np.uint8), host(c), host(l.double()),
                    host(u.double()), np.ones(n, dtype=np.uint8))


def _lp(family, m, seed):
    if family == "relaxation":
        return lpgen.mip_relaxation(seed, m=m, n=2 * m, density=min(1.0, 4.0 / m))
    if family == "energy":
        return lpgen.energy_system(seed=seed, hours=m)
    return _cover(seed, m)


def _batch_lps(case, seed):
    r = random.Random(case["count"])  # the sizes belong to the case, the LPs to the seed
    return [_cover(seed * 1000 + k, r.randint(case["mmin"], case["mmax"]), fixed=True)
            for k in range(case["count"])]


def _labels(lp, seed):
    """Training targets with the look of a covering LP's solution: most columns at 0, the others
    spread over [0, 1]; duals of the size of the costs."""
    r = np.random.default_rng(seed)
    x = np.where(r.random(lp.n) < 0.2, r.random(lp.n), 0.0)
    return x, r.random(lp.m) * 20.0


def _params(case):
    kw = dict(tol=1e-14, iter_limit=case["iters"], precision=case["precision"],
              persistent=case.get("persistent", 0))
    if not case.get("adaptive"):
        kw.update(adaptive_step=0, fixed_eta=0.9)
    return P.default_params(**kw)


def prepare(case, seed):
    seed = int(seed) % (1 << 30) + 1
    s = {"case": case}
    if case["kind"] == "solve":
        lp = _lp(case["family"], case["m"], seed)
        s["prm"] = _params(case)
        if case["start"] == "learned":
            s["model"] = P.GnnModel(seed=7)
        s["lp"] = lp if case["api"] == "host" else P.DeviceLP(lp)
    elif case["kind"] == "batch":
        s["prm"] = _params(case)
        s["lps"] = [P.DeviceLP(lp) for lp in _batch_lps(case, seed)]
    else:
        s["model"] = P.GnnModel(seed=7)
        lps = [_cover(seed * 16 + k, case["m"]) for k in range(case.get("graphs", 1))]
        s["graphs"] = [s["model"].graph(lp) for lp in lps]
        if case["kind"] == "gradient":
            for k, (g, lp) in enumerate(zip(s["graphs"], lps)):
                g.set_labels(*_labels(lp, seed * 16 + k))
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "forward":
        x, y, _ = s["model"].forward(s["graphs"][0])
        return {"x": x.astype(np.float32), "y": y.astype(np.float32)}  # a float32 network
    if case["kind"] == "gradient":
        s["model"].zero_grad()
        w = 1.0 / len(s["graphs"])
        loss = [s["model"].backward(g, w) for g in s["graphs"]]
        return {"grad": s["model"].grad(), "loss": np.array(loss, dtype=np.float32)}
    f32 = case["precision"] != "fp64"
    if case["kind"] == "batch":
        xs, ys, _ = P.pdlp_solve_batch_device(s["lps"], s["prm"])
        x, y = torch.cat(xs), torch.cat(ys)
        return {"x": x.float() if f32 else x, "y": y.float() if f32 else y}
    if case["api"] == "device":
        x, y, _ = P.pdlp_solve_device(s["lp"], s["prm"])
        return {"x": x.float() if f32 else x, "y": y.float() if f32 else y}
    if case["start"] == "learned":
        x, y, _, _ = P.pdlp_solve_warm(s["model"], s["lp"], s["prm"])
    else:
        x, y, _ = P.pdlp_solve(s["lp"], s["prm"])
    return {"x": x.astype(np.float32) if f32 else x, "y": y.astype(np.float32) if f32 else y}


# ---------------------------------------------------------------- what a pass cannot do without
def _sizes(case):
    """Rows, columns and nonzeros (expected) of a case's LP, or of all its LPs."""
    if case["kind"] == "batch":
        m = case["count"] * (case["mmin"] + case["mmax"]) / 2
        return m, 4 * m, 27 * m
    m = case["m"]
    if case["kind"] != "solve":
        k = case.get("graphs", 1)
        return m * k, 4 * m * k, 27 * m * k
    if case["family"] == "relaxation":
        return m, 2 * m, 8 * m
    if case["family"] == "energy":
        return 240 * m, 280 * m + 120, 900 * m
    return m, 4 * m, 27 * m


def work(case):
    """Inputs read once and outputs written once, plus, for every iteration, the step data of
    problems beyond L2 (a smaller problem's stays on the chip); operations of the two products
    of each step, of the KKT passes, of the network's layers."""
    m, n, z = _sizes(case)
    io = 12 * z + 8 * (m + 1) + 9 * m + 24 * n + 8 * (m + n)
    if case["kind"] in ("forward", "gradient"):
        passes = 1 if case["kind"] == "forward" else 3
        rows = 256 * (m + n)  # a hidden row: 64 float32 values
        return {"bytes": 12 * z * 6 * passes + rows * 13 * passes,
                "flops": passes * 3 * (2 * 128 * 64 * (m + n) + 4 * 64 * z)}
    it, f64 = case["iters"], case["precision"] == "fp64"
    e = 8 if f64 else 4
    v = 0 if case["precision"] == "bf16" and case.get("family") != "relaxation" else e
    step = 2 * z * (4 + v) + 4 * (m + n) + e * (10 * n + 7 * m)
    stream = it * step if step > 128e6 else 0
    return {"bytes": io + stream, "flops": it * (6 * z + 12 * (m + n)) + it / 64 * 12 * z}


# ---------------------------------------------------------------- the same in 64 bits
def _sparse(ptr, col, val, m, n):
    return torch.sparse_csr_tensor(ptr, col.long(), val, (m, n))


class _Exact:
    """Restarted PDHG with the step rules of the cases above, in float64 torch operations."""

    def __init__(self, lp):
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
        self.m, self.n = lp.m, lp.n
        ptr, col = t(lp.row_ptr), t(lp.col).long()
        self.row = torch.repeat_interleave(torch.arange(lp.m, device=DEV), ptr[1:] - ptr[:-1])
        self.col, self.ptr = col, ptr
        sense = t(lp.sense)
        self.s = torch.where(sense == lpgen.SENSE_LE, -1.0, 1.0).double()
        self.eq = sense == lpgen.SENSE_EQ
        self.val = self.s[self.row] * t(lp.val)
        self.q = self.s * t(lp.b)
        self.c, self.l, self.u = t(lp.c), t(lp.l), t(lp.u)
        order = torch.argsort(col * lp.m + self.row)
        self.torder = order
        self.tptr = torch.zeros(lp.n + 1, dtype=torch.int64, device=DEV)
        self.tptr[1:] = torch.cumsum(torch.bincount(col, minlength=lp.n), 0)
        self.k, self.kt = self.pair(self.val)

    def pair(self, val):
        return (_sparse(self.ptr, self.col, val, self.m, self.n),
                _sparse(self.tptr, self.row[self.torder], val[self.torder], self.n, self.m))

    def scaling(self):
        dr, dc = torch.ones_like(self.q), torch.ones_like(self.c)
        a = self.val.abs()
        for it in range(11):
            v = dr[self.row] * a * dc[self.col]
            how = "amax" if it < 10 else "sum"
            r = torch.zeros_like(dr).scatter_reduce(0, self.row, v, how)
            c = torch.zeros_like(dc).scatter_reduce(0, self.col, v, how)
            dr = dr / torch.where(r > 0, r.sqrt(), torch.ones_like(r))
            dc = dc / torch.where(c > 0, c.sqrt(), torch.ones_like(c))
        return dr, dc

    def dual(self, y):
        return torch.where(self.eq, y, y.clamp(min=0))

    def kkt(self, k, kt, q, c, l, u, x, y):
        rp = q - k @ x
        rp = torch.where(self.eq, rp, rp.clamp(min=0))
        lam = c - kt @ y
        up, dn = lam.clamp(min=0), (-lam).clamp(min=0)
        zero = torch.zeros_like(lam)
        rd = torch.where(torch.isinf(l), up, zero) + torch.where(torch.isinf(u), dn, zero)
        pobj = float(c @ x)
        dobj = float(q @ y + torch.where(torch.isinf(l), zero, l * up).sum()
                     - torch.where(torch.isinf(u), zero, u * dn).sum())
        nrp, nrd, gap = float(rp.norm()), float(rd.norm()), abs(pobj - dobj)
        return nrp, nrd, gap, max(nrp / (1 + float(q.norm())), nrd / (1 + float(c.norm())),
                                  gap / (1 + abs(pobj) + abs(dobj)))

    def solve(self, iters, adaptive, start=None, hint=None):
        dr, dc = self.scaling()
        k, kt = self.pair(dr[self.row] * self.val * dc[self.col])
        c, q, l, u = dc * self.c, dr * self.q, self.l / dc, self.u / dc
        box = lambda v: torch.minimum(torch.maximum(v, l), u)
        into = lambda p: (box(p[0] / dc), self.dual(self.s * p[1] / dr))
        x, y = into(start) if start else (box(torch.zeros_like(c)), torch.zeros_like(q))
        pair = [float(v.norm()) for v in (into(hint)[::-1] if hint else (c, q))]
        om = pair[0] / pair[1] if min(pair) > 1e-10 else 1.0
        eta = 1.0 / float(k.values().abs().max()) if adaptive else 0.9
        metric = lambda a: math.sqrt(om * a[0] ** 2 + a[1] ** 2 / om + a[2] ** 2)
        scaled = lambda xs, ys: self.kkt(k, kt, q, c, l, u, xs, ys)
        clip = lambda v: torch.minimum(torch.maximum(dc * v, self.l), self.u)
        plain = lambda xs, ys: self.kkt(self.k, self.kt, self.q, self.c, self.l, self.u, clip(xs),
                                        dr * ys)[3]
        xl, yl, kl, prev, since = x, y, scaled(x, y), math.inf, 0
        sx, sy, sw = torch.zeros_like(x), torch.zeros_like(y), 0.0
        it = att = 0
        while it < iters:
            att += 1
            xn = box(x - (eta / om) * (c - kt @ y))
            yn = self.dual(y + eta * om * (q - k @ (2 * xn - x)))
            used = eta
            if adaptive:
                dx, dy = xn - x, yn - y
                den = 2 * abs(float(dy @ (k @ dx)))
                bar = (om * float(dx @ dx) + float(dy @ dy) / om) / den if den > 0 else math.inf
                eta = min((1 - (att + 1) ** -0.3) * bar, (1 + (att + 1) ** -0.6) * eta)
                if used > bar:
                    continue
            x, y, it = xn, yn, it + 1
            sx, sy, sw = sx + used * x, sy + used * y, sw + used
            if it % 64 and it < iters:
                continue
            xa, ya = sx / sw, sy / sw
            if it == iters:
                if plain(xa, ya) < plain(x, y):
                    x, y = xa, ya
            if it % 64 or it == iters:
                continue
            kc, ka = scaled(x, y), scaled(xa, ya)
            ua = metric(ka) < metric(kc)
            cand, kk = ((xa, ya), ka) if ua else ((x, y), kc)
            mc, ml = metric(kk), metric(kl)
            if mc <= 0.2 * ml or (mc <= 0.8 * ml and mc > prev) or it - since >= 0.36 * it:
                ddx, ddy = float((cand[0] - xl).norm()), float((cand[1] - yl).norm())
                if ddx > 1e-10 and ddy > 1e-10:
                    om = math.exp(0.5 * math.log(ddy / ddx) + 0.5 * math.log(om))
                x, y = cand
                xl, yl, kl, prev, since = x, y, kk, math.inf, it
                sx, sy, sw = torch.zeros_like(x), torch.zeros_like(y), 0.0
            else:
                prev = mc
        return clip(x), self.s * (dr * y)


class _ExactNet:
    """The learned start's network (include/gnn.h) in float64 torch operations."""

    def __init__(self, theta, lp):
        self.e = e = _Exact(lp)
        t = torch.from_numpy(theta).to(DEV).bfloat16().double()  # the weights the passes use
        self.shapes = [("wvi", 6, 64), ("bvi", 64), ("wci", 5, 64), ("bci", 64)]
        for k in range(3):
            self.shapes += [(f"cc{k}", 64, 64), (f"cv{k}", 64, 64), (f"bc{k}", 64),
                            (f"vv{k}", 64, 64), (f"vc{k}", 64, 64), (f"bv{k}", 64)]
        self.shapes += [("wx", 64), ("bx", 1), ("wy", 64), ("by", 1)]
        self.p, o = {}, 0
        for name, *sh in self.shapes:
            self.p[name] = t[o:o + math.prod(sh)].reshape(sh)
            o += math.prod(sh)
        val = e.s[e.row] * e.val  # the caller's signs
        dr = (e.ptr[1:] - e.ptr[:-1]).double()
        dc = (e.tptr[1:] - e.tptr[:-1]).double()
        sq = lambda i, k: torch.zeros(k, dtype=torch.float64, device=DEV).index_add(0, i, val * val).sqrt()
        nr, nc = sq(e.row, e.m), sq(e.col, e.n)
        self.cmax = float(e.c.abs().max())
        slog = lambda v: v.sign() * torch.log1p(v.clamp(-1e3, 1e3).abs())
        one = torch.ones_like
        fv = [e.c / self.cmax, slog(e.l), slog(e.u), nc / nc.max(), dc / dc.max(), one(e.c)]
        fc = [e.s * e.q / e.q.abs().max(), torch.where(e.eq, 0.0, e.s), nr / nr.max(),
              dr / dr.max(), one(e.q)]
        # the features are float32 arrays
        self.fv, self.fc = (torch.stack(f, 1).float().double() for f in (fv, fc))
        wr, wc = val / dr.clamp(min=1)[e.row], val / dc.clamp(min=1)[e.col]
        self.R, self.Rt = e.pair(wr)
        self.C, self.Ct = e.pair(wc)

    def forward(self):
        p = self.p
        hv, hc = [(self.fv @ p["wvi"] + p["bvi"]).relu()], [(self.fc @ p["wci"] + p["bci"]).relu()]
        sc, sv = [], []
        for k in range(3):
            sc.append(self.R @ hv[-1])
            hc.append((hc[-1] @ p[f"cc{k}"] + sc[-1] @ p[f"cv{k}"] + p[f"bc{k}"]).relu())
            sv.append(self.Ct @ hc[-1])
            hv.append((hv[-1] @ p[f"vv{k}"] + sv[-1] @ p[f"vc{k}"] + p[f"bv{k}"]).relu())
        self.zx, self.zy = hv[-1] @ p["wx"] + p["bx"], hc[-1] @ p["wy"] + p["by"]
        self.hv, self.hc, self.sc, self.sv = hv, hc, sc, sv
        return (self.e.l + (self.e.u - self.e.l) * torch.sigmoid(self.zx),
                torch.nn.functional.softplus(self.zy))

    def gradient(self, xs, ys):
        """(gradient, loss) of a boxed LP without equality rows."""
        x, y = self.forward()
        p, hv, hc, sc, sv = self.p, self.hv, self.hc, self.sc, self.sv
        w = self.e.u - self.e.l
        w = torch.where(w > 0, w, torch.ones_like(w))
        ex, ey = (x - xs) / w, y - ys / self.cmax
        s = torch.sigmoid(self.zx)
        dzx = 2.0 / self.e.n * ex / w * (self.e.u - self.e.l) * s * (1 - s)
        dzy = 2.0 / self.e.m * ey * torch.sigmoid(self.zy)
        g = {"wx": hv[-1].T @ dzx, "bx": dzx.sum()[None], "wy": hc[-1].T @ dzy, "by": dzy.sum()[None]}
        dv, dc = dzx[:, None] * p["wx"], dzy[:, None] * p["wy"]
        for k in (2, 1, 0):
            d = dv * (hv[k + 1] > 0)
            g[f"vv{k}"], g[f"vc{k}"], g[f"bv{k}"] = hv[k].T @ d, sv[k].T @ d, d.sum(0)
            dv = d @ p[f"vv{k}"].T
            d = (dc + self.C @ (d @ p[f"vc{k}"].T)) * (hc[k + 1] > 0)
            g[f"cc{k}"], g[f"cv{k}"], g[f"bc{k}"] = hc[k].T @ d, sc[k].T @ d, d.sum(0)
            dc = d @ p[f"cc{k}"].T
            dv = dv + self.Rt @ (d @ p[f"cv{k}"].T)
        d = dv * (hv[0] > 0)
        g["wvi"], g["bvi"] = self.fv.T @ d, d.sum(0)
        d = dc * (hc[0] > 0)
        g["wci"], g["bci"] = self.fc.T @ d, d.sum(0)
        loss = float((ex * ex).mean() + (ey * ey).mean())
        return torch.cat([g[name].reshape(-1) for name, *_ in self.shapes]), loss


def exact(case, seed):
    seed = int(seed) % (1 << 30) + 1
    if case["kind"] == "solve":
        lp = _lp(case["family"], case["m"], seed)
        e = _Exact(lp)
        start = hint = None
        if case["start"] == "learned":
            net = _ExactNet(P.GnnModel(seed=7).params(), lp)
            x, y = net.forward()
            hint = torch.minimum(torch.maximum(x, e.l), e.u), net.cmax * y
            at = lambda z: e.kkt(e.k, e.kt, e.q, e.c, e.l, e.u, *z)[3]
            cold = torch.zeros_like(x).clamp(e.l, e.u), torch.zeros_like(y)
            start = hint if at(hint) < at(cold) else None
        x, y = e.solve(case["iters"], case["adaptive"], start, hint)
        return {"x": x, "y": y}
    if case["kind"] == "batch":
        both = [_Exact(lp).solve(case["iters"], False) for lp in _batch_lps(case, seed)]
        return {"x": torch.cat([b[0] for b in both]), "y": torch.cat([b[1] for b in both])}
    theta = P.GnnModel(seed=7).params()
    lps = [_cover(seed * 16 + k, case["m"]) for k in range(case.get("graphs", 1))]
    if case["kind"] == "forward":
        net = _ExactNet(theta, lps[0])
        x, y = net.forward()
        return {"x": x, "y": net.cmax * y}
    got = []
    for k, lp in enumerate(lps):
        xs, ys = (torch.from_numpy(v).to(DEV) for v in _labels(lp, seed * 16 + k))
        got.append(_ExactNet(theta, lp).gradient(xs, ys))
    return {"grad": sum(g for g, _ in got) / len(got), "loss": torch.tensor([v for _, v in got])}
