"""The work this library is timed on: what a user of it calls, over the sizes it is used at.

Every case is a weighted least-squares problem of the SPI sky-and-background model (19 detectors,
a 5 x 5 dither raster, sources cut into time-bins, one background column per pointing, 19
detector-pattern columns per block of pointings, optionally a grid of sky pixels), the family the
tests and the benchmark use.  The geometry (which column meets which row) comes from the case; the
responses, the counts and so all values come from the seed, and are made on the GPU.
"""
import functools
import math
import types

import numpy as np
import torch

import paper_1305_5683_gb300 as spi

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")
ND = 19          # detectors: rows per pointing
RASTER = 5       # dither raster
WINDOW = 64      # pointings handled at a time by the input maker


def _case(name, call, precision, P, sources, lo, hi, det, **more):
    return dict(name=name, call=call, precision=precision, P=P, sources=sources, lo=lo, hi=hi, det=det,
                geometry=0, **more)


def listed():
    return [
        # a quick look at one short observation: factor, solution and every variance; launches and
        # host calls are all that counts
        _case("fp64-step-P300", "step", "fp64", 300, 40, 10, 300, 100),
        # an ordinary observation of a few days, an odd number of pointings
        _case("fp64-step-P2003", "step", "fp64", 2003, 50, 20, 200, 125),
        # many short independent observations as one forest, sizes ragged (P log-uniform 50-2,000)
        _case("fp64-forest-48", "forest", "fp64", 2000, 0, 0, 0, 0, count=48),
        # the large observation: new values on the same pattern (a band, a Newton step), solution only
        _case("fp64-refit-P20000", "refit", "fp64", 20000, 500, 20, 2000, 500),
        # further right-hand sides on a kept factor (bootstrap, model trials)
        _case("fp64-solve-P20000", "solve", "fp64", 20000, 500, 20, 2000, 500),
        # the error bars of every unknown of the large observation
        _case("fp64-variances-P20000", "variances", "fp64", 20000, 500, 20, 2000, 500),
        # the same two in the mixed form (FP32 updates, FP64 pivots and refinement)
        _case("mixed-refit-P20000", "refit", "mixed", 20000, 500, 20, 2000, 500),
        _case("mixed-variances-P20000", "variances", "mixed", 20000, 500, 20, 2000, 500),
        # energy bands of one observation in one batch: factor, refined solution, every variance
        _case("mixed-bands-16-P5000", "bands", "mixed", 5000, 200, 10, 200, 500, count=16),
        # diffuse sky: one dense separator of thousands of pixels; the pixels' variances
        _case("mixed-sky-P4000", "step", "mixed", 4000, 100, 10, 1000, 500, pix=1.0),
        # the step before the solver: N = H^T W H and b from the design matrix on the device
        _case("fp64-assemble-P5000", "assemble", "fp64", 5000, 200, 10, 200, 500),
        # covariances of the time-bins of one stretch of the observation
        _case("fp64-covariance-P5000", "covariance", "fp64", 5000, 200, 10, 200, 500, count=512),
    ]


def draw(rng):
    """A case of the same ranges: any call, sizes spread over their logarithm, odd ones among them."""
    call = rng.choice(["step", "step", "sky", "refit", "solve", "variances", "bands", "forest", "assemble",
                       "covariance"])
    mixed = rng.random() < 0.5
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    geometry = rng.randrange(1, 1000)
    top = {"step": 12000, "sky": 3500, "refit": 20000, "solve": 20000, "variances": 12000, "bands": 4000,
           "forest": 1500, "assemble": 6000, "covariance": 6000}[call]
    P = logint(60 if call != "sky" else 400, top)
    c = dict(call="step" if call == "sky" else call, precision="mixed" if mixed else "fp64", P=P,
             sources=max(5, P // 40), lo=max(5, P // 1000), hi=max(10, P // 10), det=max(25, min(500, P // 4)),
             geometry=geometry)
    if call == "sky":
        c.update(pix=round(rng.uniform(1.2, 3.0), 2), sources=max(5, P // 60))
    if call == "forest":
        c.update(precision="fp64", count=logint(2, 40))
    if call == "bands":
        c.update(precision="mixed", count=logint(2, 16))
    if call in ("assemble", "covariance"):
        c.update(precision="fp64")
    if call == "covariance":
        c.update(count=logint(8, 512))
    return c


# ---------------------------------------------------------------------------------- the model
def _angle(lon1, lat1, lon2, lat2):
    l1, b1, l2, b2 = (np.radians(v) for v in (lon1, lat1, lon2, lat2))
    s = np.sin((b2 - b1) / 2) ** 2 + np.cos(b1) * np.cos(b2) * np.sin((l2 - l1) / 2) ** 2
    return np.degrees(2 * np.arcsin(np.sqrt(np.clip(s, 0.0, 1.0))))


class Geometry:
    """Which columns of the design matrix meet which pointings."""

    def __init__(self, P, sources, lo, hi, det, pix, seed):
        rng = np.random.default_rng(seed)
        sky = pix > 0
        half = 35.0 if sky else 20.0
        lon, lat = rng.uniform(-half, half, sources), rng.uniform(-half, half, sources)
        nq = RASTER * RASTER
        off = np.arange(nq)
        plon, plat = 2.0 * (off % RASTER - RASTER // 2), 2.0 * (off // RASTER - RASTER // 2)
        self.pos = np.arange(P) % nq
        if sky:  # 7 x 7 targets 10 deg apart, each visited for one raster
            t = np.arange(49)
            plon = (((t % 7) - 3) * 10.0)[:, None] + plon[None, :]
            plat = (((t // 7) - 3) * 10.0)[:, None] + plat[None, :]
            plon, plat = plon.ravel(), plat.ravel()
            self.pos = ((np.arange(P) // nq) % 49) * nq + np.arange(P) % nq
        npos = len(plon)
        vis = _angle(lon[:, None], lat[:, None], plon[None, :], plat[None, :]) < 15.0
        start, end, src = [], [], []
        for s in range(sources):
            edges = [0]
            while edges[-1] < P:
                edges.append(min(P, edges[-1] + max(1, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))))
            if len(edges) > 2 and edges[-1] - edges[-2] < lo:
                edges.pop(-2)
            for a, b in zip(edges[:-1], edges[1:]):
                if vis[s, np.unique(self.pos[a:b])].any():
                    start.append(a), end.append(b), src.append(s)
        order = np.lexsort((src, start))
        self.start, self.end, self.src = (np.array(v, np.int64)[order] for v in (start, end, src))
        nblk = max(1, P // det + (1 if P % det >= (det + 1) // 2 else 0))
        self.block = np.minimum(np.arange(P) // det, nblk - 1)
        self.pvis = np.zeros((0, npos), bool)
        if sky:
            k = int(round(70.0 / pix))
            grid = (np.arange(k) + 0.5) * pix - 35.0
            pvis = _angle(np.tile(grid, k)[:, None], np.repeat(grid, k)[:, None], plon[None, :], plat[None, :]) < 15.0
            self.pvis = pvis[pvis[:, np.unique(self.pos)].any(axis=1)]
        self.P, self.npos, self.sources, self.vis = P, npos, sources, vis
        self.ndet, self.nbin, self.nsky = nblk * ND, len(self.start), len(self.pvis)
        self.nrest = self.ndet + self.nbin + self.nsky   # all columns but the pointings'
        self.n = P + self.nrest
        self.pattern = None

    def windows(self):
        """(first pointing, last + 1, detector-block columns, bins, pixels) of each stretch of pointings."""
        for p0 in range(0, self.P, WINDOW):
            p1 = min(self.P, p0 + WINDOW)
            bins = np.nonzero((self.start < p1) & (self.end > p0))[0]
            pix = np.nonzero(self.pvis[:, np.unique(self.pos[p0:p1])].any(axis=1))[0]
            yield p0, p1, np.arange(self.block[p0] * ND, (self.block[p1 - 1] + 1) * ND), bins, pix


def _up(a):
    return torch.as_tensor(a, device=DEV)


class Draw:
    """The values of one seed on one geometry: D (the pointings' diagonal), B (pointings x the others, by
    window), C (the others, dense, upper triangle), b; N = [[D, B], [B', C]]."""

    def __init__(self, geo, seed, scale=None, keep_rows=False):
        gen = torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFF)
        def uni(lo, hi, *shape):
            return lo + (hi - lo) * torch.rand(*shape, dtype=torch.float64, device=DEV, generator=gen)
        P, f64 = geo.P, dict(dtype=torch.float64, device=DEV)
        u, g, h = uni(50, 200, ND), uni(0.8, 1.2, P, ND), uni(0.8, 1.2, P, ND)
        resp = uni(0.1, 1.0, geo.sources, geo.npos, ND)
        if scale is not None:
            resp = resp * scale[:, None, None]
        xp = uni(0.9, 1.1, P)
        xr = torch.cat([uni(0, 5, geo.ndet), uni(0, 20, geo.nbin), uni(0, 5, geo.nsky)])
        used = np.unique(geo.pos)
        sky = uni(0.1, 1.0, geo.nsky, len(used), ND) if geo.nsky else None
        at = np.searchsorted(used, geo.pos)
        src, start, end, pos, block = (_up(v) for v in (geo.src, geo.start, geo.end, geo.pos, geo.block))
        vis, pvis, at = _up(geo.vis), _up(geo.pvis), _up(at)
        dd = torch.arange(ND, device=DEV)
        self.geo, self.D, self.B = geo, torch.empty(P, **f64), []
        self.C, self.b = torch.zeros(geo.nrest, geo.nrest, **f64), torch.zeros(geo.n, **f64)
        self.rows = []
        for p0, p1, dets, bins, pix in geo.windows():
            m, p = p1 - p0, torch.arange(p0, p1, device=DEV)
            bt, xt = _up(bins), _up(pix)
            cols = torch.cat([_up(dets), geo.ndet + bt, geo.ndet + geo.nbin + xt])
            A = torch.zeros(m, ND, len(cols), **f64)
            A[(p - p0)[:, None], dd[None, :], (block[p] - int(geo.block[p0]))[:, None] * ND + dd[None, :]] = h[p0:p1]
            on = (start[bt][None, :] <= p[:, None]) & (p[:, None] < end[bt][None, :]) & vis[src[bt]][:, pos[p]].T
            A[:, :, len(dets):len(dets) + len(bins)] = (resp[src[bt][None, :], pos[p][:, None]] * on[:, :, None]).transpose(1, 2)
            if len(pix):
                on = pvis[xt][:, pos[p]].T
                A[:, :, len(dets) + len(bins):] = (sky[xt[None, :], at[p][:, None]] * on[:, :, None]).transpose(1, 2)
            a = u[None, :] * g[p0:p1]                       # the pointing columns' entries
            y = torch.poisson(a * xp[p0:p1, None] + A @ xr[cols], generator=gen)
            w = 1.0 / torch.clamp(y, min=1.0)
            W = A * w[:, :, None]
            flat = A.reshape(m * ND, -1)
            self.C[cols[:, None], cols[None, :]] += flat.T @ W.reshape(m * ND, -1)
            self.D[p0:p1] = (a * a * w).sum(1)
            self.B.append((cols, torch.einsum("pd,pdc->pc", a, W)))
            self.b[p0:p1] = (a * w * y).sum(1)
            self.b[P + cols] += flat.T @ (w * y).reshape(-1)
            if keep_rows:
                full = torch.cat([torch.diag_embed(a.T).permute(1, 0, 2), A], dim=2).reshape(m * ND, -1)
                r, c = torch.nonzero(full, as_tuple=True)
                ids = torch.cat([p, P + cols])
                self.rows.append((torch.bincount(r, minlength=m * ND), ids[c], full[r, c], w.reshape(-1), y.reshape(-1)))

    def csc(self):
        """(colptr, rowind, values) of N's lower triangle; the pattern is the geometry's alone."""
        geo = self.geo
        if geo.pattern is None:   # every stored product is a sum of positive terms
            count, rows = [], []
            for (cols, B), (p0, p1, *_) in zip(self.B, geo.windows()):
                on = torch.cat([torch.ones(p1 - p0, 1, dtype=torch.bool, device=DEV), B > 0], dim=1)
                ids = torch.cat([torch.arange(p0, p1, device=DEV)[:, None], (geo.P + cols)[None, :].expand(p1 - p0, -1)], dim=1)
                count.append(on.sum(1)), rows.append(ids[on])
            where = []
            for j in range(0, geo.nrest, 2048):
                part = torch.triu(self.C[j:j + 2048], diagonal=j)
                r, c = torch.nonzero(part, as_tuple=True)
                count.append(torch.bincount(r, minlength=len(part)))
                rows.append(geo.P + c), where.append((r + j) * geo.nrest + c)
            colptr = np.concatenate([[0], torch.cumsum(torch.cat(count), 0).cpu().numpy()]).astype(np.int64)
            geo.pattern = colptr, torch.cat(rows).to(torch.int32).cpu().numpy(), torch.cat(where)
        colptr, rowind, where = geo.pattern
        lead = []
        for (_, B), (p0, p1, *_) in zip(self.B, geo.windows()):
            full = torch.cat([self.D[p0:p1, None], B], dim=1)
            lead.append(full[full > 0])
        return colptr, rowind, torch.cat(lead + [self.C.view(-1)[where]])

    def solved(self, need):
        """x, diag(N^-1) and the inverse of the others' Schur complement, dense, in 64 bits."""
        P, D, b = self.geo.P, self.D, self.b
        S = torch.triu(self.C)
        S = S + torch.triu(S, 1).T
        t = b[P:].clone()
        for (cols, B), (p0, p1, *_) in zip(self.B, self.geo.windows()):
            S[cols[:, None], cols[None, :]] -= B.T @ (B / D[p0:p1, None])
            t[cols] -= B.T @ (b[p0:p1] / D[p0:p1])
        L = torch.linalg.cholesky(S)
        del S
        x = torch.empty_like(b)
        x[P:] = torch.cholesky_solve(t[:, None], L)[:, 0]
        inv = torch.cholesky_inverse(L) if need else None
        del L
        v = torch.empty_like(b)
        if need:
            v[P:] = torch.diagonal(inv)
        for (cols, B), (p0, p1, *_) in zip(self.B, self.geo.windows()):
            x[p0:p1] = (b[p0:p1] - B @ x[P + cols]) / D[p0:p1]
            if need:
                E = B / D[p0:p1, None]
                v[p0:p1] = 1.0 / D[p0:p1] + (E * (E @ inv[cols[:, None], cols[None, :]])).sum(1)
        return x, v, inv


@functools.lru_cache(maxsize=2)
def _geometries(P, sources, lo, hi, det, pix, geometry, members):
    if not members:
        return (Geometry(P, sources, lo, hi, det, pix, geometry),)
    rng, got = np.random.default_rng(1_000_003 + geometry), []
    for i in range(members):   # sizes of a forest: P log-uniform from 50 up
        p = int(round(math.exp(rng.uniform(math.log(50), math.log(max(51, P))))))
        got.append(Geometry(p, max(5, p // 10), max(5, p // 40), max(6, p // 2), max(25, p // 4), 0.0, i))
    return tuple(got)


def _geo(case):
    members = case["count"] if case["call"] == "forest" else 0
    return _geometries(case["P"], case["sources"], case["lo"], case["hi"], case["det"], case.get("pix", 0.0),
                       case["geometry"], members)


def _draws(case, seed):
    geos = _geo(case)
    if case["call"] == "bands":   # one pattern; the sources' spectra and the counts differ from band to band
        rng = np.random.default_rng(seed)
        slope = rng.uniform(1.5, 3.0, geos[0].sources)
        energy = np.exp(np.linspace(0.0, math.log(50.0), case["count"]))
        for k, e in enumerate(energy):
            yield Draw(geos[0], seed * 1009 + k, scale=_up(e ** -slope))
    else:
        for k, geo in enumerate(geos):
            yield Draw(geo, seed * 1009 + k, keep_rows=case["call"] == "assemble")


def _chosen(case):
    """The indices asked for: sky pixels, or the time-bins of one stretch; None for every unknown."""
    geo = _geo(case)[0]
    if case.get("pix"):
        return np.arange(geo.n - geo.nsky, geo.n, dtype=np.int32)
    if case["call"] == "covariance":
        m = min(case["count"], geo.nbin)
        first = (geo.nbin - m) // 2
        return np.arange(geo.P + geo.ndet + first, geo.P + geo.ndet + first + m, dtype=np.int32)
    return None


# ---------------------------------------------------------------------------------- the calls
def prepare(case, seed):
    """The program's data on the GPU and a context that has served one earlier set of values."""
    call = case["call"]
    values, b, probs, rows = [], [], [], None
    for d in _draws(case, seed):
        colptr, rowind, v = d.csc()
        values.append(v), b.append(d.b)
        probs.append(types.SimpleNamespace(n=d.geo.n, colptr=colptr, rowind=rowind))
        rows = d.rows
        del d
    precision = spi.SPI_PREC_MIXED_FP32 if case["precision"] == "mixed" else spi.SPI_PREC_FP64
    values, b = torch.cat(values), torch.cat(b)
    st = types.SimpleNamespace(call=call, values=values, b=b, n=probs[0].n, x=torch.empty_like(b), idx=None)
    if call == "forest":
        st.s = spi.Solver.for_problems(probs, precision=precision)
    elif call == "bands":
        st.s = spi.Solver.for_problem(probs[0], precision=precision, batch=case["count"])
    else:
        st.s = spi.Solver.for_problem(probs[0], precision=precision)
    if call == "assemble":
        count, col, val, w, y = (torch.cat(v) for v in zip(*rows))
        ptr = np.concatenate([[0], torch.cumsum(count, 0).cpu().numpy()])
        st.s.normal_setup((np.ones(len(val)), col.cpu().numpy().astype(np.int32), ptr))
        st.h, st.w, st.y, st.out = val, w, y, torch.empty_like(values)
        return st
    idx = _chosen(case)
    st.idx = None if idx is None else _up(idx)
    m = len(b) if idx is None else len(idx)
    st.var = torch.empty((m, m) if call == "covariance" else m, dtype=torch.float64, device=DEV)
    (st.s.factor_batch if call == "bands" else st.s.factor)(values * 1.25)
    if call in ("solve", "variances", "covariance"):
        st.s.factor(values)
    if call != "covariance":
        keep, st.values = st.values, st.values * 1.25
        run(st)
        st.values = keep
    if call in ("solve", "variances"):
        st.s.factor(values)
    return st


def run(st):
    s, call = st.s, st.call
    if call in ("step", "forest"):
        s.factor(st.values)
        s.solve(st.b, st.x)
        s.diag_inverse(st.idx, st.var)
        return {"x": st.x, "var": st.var}
    if call == "refit":
        s.factor(st.values)
        return {"x": s.solve(st.b, st.x)}
    if call == "solve":
        return {"x": s.solve(st.b, st.x)}
    if call == "variances":
        return {"var": s.diag_inverse(None, st.var)}
    if call == "bands":
        s.factor_batch(st.values)
        s.solve_batch(st.b, st.x)
        s.diag_inverse_batch(out=st.var)
        return {"x": list(st.x.view(-1, st.n)), "var": list(st.var.view(-1, st.n))}
    if call == "covariance":
        return {"cov": s.inverse_block(st.idx, st.var)}
    s.normal_assemble(st.h, st.w, st.y, st.out, st.x)
    return {"values": st.out, "b": st.x}


def exact(case, seed):
    """The same from dense 64-bit algebra: pointings eliminated by hand, a dense Cholesky of the rest."""
    call, idx = case["call"], _chosen(case)
    xs, vs = [], []
    for k, d in enumerate(_draws(case, seed)):
        if call == "assemble":
            return {"values": d.csc()[2], "b": d.b}
        if call == "bands" and k >= 2:   # two bands tell; all would take minutes
            break
        x, v, inv = d.solved(call not in ("refit", "solve"))
        if call == "covariance":
            at = _up(idx.astype(np.int64)) - d.geo.P
            return {"cov": inv[at[:, None], at[None, :]]}
        xs.append(x), vs.append(v if idx is None else v[_up(idx.astype(np.int64))])
    if call == "bands":
        rest = [None] * (case["count"] - len(xs))
        return {"x": xs + rest, "var": vs + rest}
    x, v = torch.cat(xs), torch.cat(vs)
    return {"refit": {"x": x}, "solve": {"x": x}, "variances": {"var": v}}.get(call, {"x": x, "var": v})


@functools.lru_cache(maxsize=16)
def _counts(key):
    """(n, entries of N, entries of L, factor flops, all variances' flops, largest front, entries of H)."""
    case, total, h = dict(key), np.zeros(6), 0.0
    for geo in _geo(case):
        d = Draw(geo, 0, keep_rows=case["call"] == "assemble")
        colptr, rowind, _ = d.csc()
        i = spi.Solver(geo.n, colptr, rowind).info()
        total += [geo.n, i["nnz_a"], i["nnz_l"], i["factor_flops"], i["diag_flops_all"], i["max_front"]]
        h += sum(len(r[1]) for r in d.rows)
    return (*total, h)


def work(case):
    """One pass's floor: inputs once, outputs once, the factor written (and read) once; the
    arithmetic of the exact column counts."""
    n, nnz, nnzl, ff, df, front, h = _counts(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
    word = 4.0 if case["precision"] == "mixed" else 8.0
    idx, call = _chosen(case), case["call"]
    times = case["count"] if call == "bands" else 1
    m = n if idx is None else len(idx)
    diag = df if idx is None else (m ** 3 / 3.0 if case.get("pix") else df * m / n)
    if call == "assemble":   # each row's lower column pairs: a multiply-add each, and the weight's product
        rows = ND * case["P"]
        return {"bytes": 8.0 * (h + 2 * rows + nnz + n), "flops": h * (h / rows + 1) + 2 * h}
    if call == "covariance":
        return {"bytes": word * nnzl + 8.0 * m * m, "flops": diag + front * m * m}
    if call == "solve":
        return {"bytes": word * nnzl + 16.0 * n, "flops": 4.0 * nnzl}
    if call == "variances":
        return {"bytes": word * nnzl + 8.0 * n, "flops": diag}
    flops, nbytes = ff + 4.0 * nnzl, 8.0 * nnz + word * nnzl + 16.0 * n
    if call != "refit":
        flops, nbytes = flops + diag, nbytes + 8.0 * m
    return {"bytes": times * nbytes, "flops": times * flops}


def tolerance(case):
    """About four times the distance from the dense 64-bit results measured over these sizes.  An x
    in 64 bits carries rounding times the condition of N (up to 4e-12 of its norm here), a variance,
    a covariance or an entry of N, all sums of squares or of positive terms, a few roundings
    (3e-15).  The mixed form's x is refined to 64-bit residuals (2e-11); its variances keep the
    32-bit factor's error (8e-7 of their norm, 1e-5 of the worst one)."""
    if case["precision"] == "mixed":
        return {"rel": 1e-10, "max": 1e-9} if case["call"] in ("refit", "solve") else {"rel": 4e-6, "max": 4e-5}
    if case["call"] in ("variances", "covariance", "assemble"):
        return {"rel": 2e-14, "max": 2e-13}
    return {"rel": 2e-11, "max": 2e-10}
