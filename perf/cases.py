"""Performance cases of the bispectrum-multipole estimator: what its users run, through the package's
public entry points (``api.Plan.estimate``, ``.graph`` / ``Graph.launch``, ``.estimate_host`` and
``api.ShellPlan.estimate``), from one 32^3 field to the 512^3 benchmark field.

A case holds the plan's parameters (grid, box, k1 bins, (mu, t) bins, l_max, precision), the number of
fields per call and the entry point.  The fields are seeded realisations of the synthetic recipe the
package's own generator documents (P(k) = A k^-2, sigma_G = 0.1, f_NG = 0.5, a Kaiser factor).  A
program builds a plan once and keeps it for all its fields, so plans are kept per set of parameters;
fields, workspaces, graphs and output buffers are made anew for every state.

Outputs.  Every call returns all of its multipoles, a list with one array per field.  The fp64 path
returns the doubles as they come; on the paths with FP32 transforms and products (fp32, mixed,
mixed_tc and the shell estimator) a program keeps its multipoles in single precision, which holds
every digit these paths resolve (their documented accuracy is 1e-4 of a bin), so they are returned as
float32.  ``exact`` says what they should be, in 64 bits.
"""
import functools
import math

import numpy as np
import torch

from paper_2405_14513_gb300 import api


# ------------------------------------------------------------------------------------------------
# The cases
def _case(name, ng, box, nk1, nmu, nt, lmax, precision="mixed_tc", batch=1, entry="estimate", lo=1.0 / 12, hi=1.0 / 3,
          log=False, grids="", beta=0.5):
    """k1 edges: nk1 bins, linear or logarithmic, from lo N_g k_f to hi N_g k_f.  grids: (mu, t) bins per
    even l (an n x n grid each), or "" for nmu x nt at every l."""
    c = {"ng": ng, "box": box, "nk1": nk1, "nmu": nmu, "nt": nt, "lmax": lmax, "precision": precision, "batch": batch,
         "entry": entry, "lo": lo, "hi": hi, "log": log, "grids": grids, "beta": beta}
    if name:
        c["name"] = name
    return c


def listed():
    kmin = 2 * math.pi / 215.0
    return [
        # one small field, the smallest call anybody makes in earnest: latency and launches
        _case("single_32", 32, 600.0, 3, 5, 5, 6),
        # a 3 x 2^k grid with the paper's logarithmic k1 bins and its per-l (mu, t) grids, a ragged batch
        _case("perl_48_x3", 48, 800.0, 6, 12, 12, 6, batch=3, log=True, grids="12,12,8,6"),
        # the 64^3 workload of the benchmark, one field per call
        _case("single_64", 64, 1000.0, 6, 5, 5, 6),
        # the same workload in FP64: how results are verified
        _case("verify_64_fp64", 64, 1000.0, 6, 5, 5, 6, precision="fp64"),
        # plain FP32, a 3 x 2^k grid, two fields, monopole and quadrupole only
        _case("plain_96_fp32_x2", 96, 750.0, 10, 10, 10, 2, precision="fp32", batch=2),
        # the default precision of a plan, one 128^3 mock
        _case("default_128_mixed", 128, 500.0, 12, 10, 10, 6, precision="mixed"),
        # many mocks: 16 fields of 128^3 per replay of a captured estimate
        _case("mocks_128_x16", 128, 500.0, 12, 10, 10, 6, batch=16, entry="graph"),
        # the 256^3 workload of the precision study, from and to host memory
        _case("study_256_host", 256, 1000.0, 20, 20, 20, 6, entry="host"),
        # a full batch of the serving loop's 256^3 plan (30 k1 bins)
        _case("serve_256_x4", 256, 1000.0, 30, 10, 10, 6, batch=4),
        # the paper's validation: 384^3, one narrow k1 bin (2.1 +- 0.1 Mpc^-1), ten realisations per call
        _case("validate_384_x10", 384, 215.0, 1, 10, 10, 6, batch=10, lo=2.0 / kmin / 384, hi=2.2 / kmin / 384, beta=1.0),
        # the benchmark's headline: one 512^3 field
        _case("headline_512", 512, 2000.0, 30, 20, 20, 6),
        # the m = 0 comparison estimator on spherical shells
        _case("shell_64", 64, 1000.0, 6, 5, 5, 6, precision="mixed", entry="shell"),
    ]


def draw(rng):
    if rng.random() < 0.06:
        ng = rng.choice([24, 32, 48, 64])
        return _case("", ng, 1000.0 * rng.uniform(0.3, 2), rng.randint(2, 8), rng.randint(2, 8), rng.randint(2, 8),
                     rng.choice([0, 2, 4, 6]), precision="mixed", entry="shell")
    precision = rng.choices(["mixed_tc", "mixed", "fp32", "fp64"], [0.64, 0.16, 0.1, 0.1])[0]
    top = {"mixed_tc": 384, "mixed": 192, "fp32": 192, "fp64": 64}[precision]
    sizes = [n for n in (16, 24, 32, 48, 64, 96, 128, 192, 256, 384) if n <= top]
    ng = rng.choice(sizes)
    batch = 1
    if precision != "fp64":
        batch = min(16, max(1, int((192.0 / ng) ** 3))) if ng < 192 else 1
        batch = max(1, round(math.exp(rng.uniform(0, math.log(batch)))))
    lo = rng.uniform(1 / 12, 1 / 5)
    hi = lo + (1 / 3 - lo) * rng.uniform(0.3, 1) if rng.random() < 0.3 else 1 / 3
    nk1 = max(1, round(math.exp(rng.uniform(0, math.log(30)))))
    lmax = rng.choice([0, 2, 4, 6, 6, 8])
    grids = ""
    if rng.random() < 0.2:
        n = rng.randint(4, 14)
        grids = ",".join(str(max(1, n - 2 * (l // 4))) for l in range(0, lmax + 1, 2))
    entry = rng.choices(["estimate", "graph", "host"], [0.6, 0.25, 0.15])[0]
    return _case("", ng, round(math.exp(rng.uniform(math.log(100), math.log(2000))), 1), nk1, rng.randint(1, 20),
                 rng.randint(1, 20), lmax, precision=precision, batch=batch, entry=entry, lo=lo, hi=hi,
                 log=rng.random() < 0.3, grids=grids, beta=rng.choice([0.5, 1.0]))


# ------------------------------------------------------------------------------------------------
# Inputs
def _edges(c):
    kf = 2.0 * math.pi / c["box"]
    lo, hi = c["lo"] * c["ng"], c["hi"] * c["ng"]
    e = (np.geomspace(lo, hi, c["nk1"] + 1) if c["log"] else np.linspace(lo, hi, c["nk1"] + 1)) * kf
    if c["hi"] == 1.0 / 3:
        e[-1] = (c["ng"] / 3.0) * kf
    return e


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _field(ng, box, seed, beta):
    """One redshift-space field delta[x][y][z], float64, z the line of sight."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    kf = 2.0 * math.pi / box
    k1 = torch.fft.fftfreq(ng, d=1.0 / ng, dtype=torch.float64, device=dev) * kf
    kz = torch.fft.rfftfreq(ng, d=1.0 / ng, dtype=torch.float64, device=dev) * kf
    k2 = k1[:, None, None] ** 2 + k1[None, :, None] ** 2 + kz[None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    w = torch.fft.rfftn(torch.randn((ng, ng, ng), generator=gen, dtype=torch.float64, device=dev))
    w *= k2.rsqrt()
    w[0, 0, 0] = 0.0
    g = torch.fft.irfftn(w, s=(ng, ng, ng), dim=(0, 1, 2))
    g *= 0.1 / g.std()
    d = g + 0.5 * (g * g - (g * g).mean())
    w = torch.fft.rfftn(d)
    w *= 1.0 + beta * kz[None, None, :] ** 2 / k2
    return torch.fft.irfftn(w, s=(ng, ng, ng), dim=(0, 1, 2))


def _fields(c, seed):
    dt = torch.float64 if c["precision"] == "fp64" else torch.float32
    out = torch.empty((c["batch"],) + (c["ng"],) * 3, dtype=dt, device=_device())
    for f in range(c["batch"]):
        out[f] = _field(c["ng"], c["box"], int(seed) * 64 + f, c["beta"])
    return out


@functools.lru_cache(maxsize=None)
def _plan(ng, box, edges, nmu, nt, lmax, precision, batch, grids):
    return api.Plan(ng, box, list(edges), nmu, nt, lmax, precision=precision, max_batch=batch,
                    mu_t_bins_l=[int(g) for g in grids.split(",")] if grids else None)


@functools.lru_cache(maxsize=None)
def _shell_plan(ng, box, edges, nmu, nt, lmax):
    return api.ShellPlan(ng, box, list(edges), nmu, nt, lmax)


def prepare(case, seed):
    c = case
    edges = tuple(float(e) for e in _edges(c))
    field = _fields(c, seed)
    if c["entry"] == "shell":
        plan = _shell_plan(c["ng"], c["box"], edges, c["nmu"], c["nt"], c["lmax"])
        return {"case": c, "plan": plan, "field": field[0].contiguous(), "ws": plan.workspace()}
    plan = _plan(c["ng"], c["box"], edges, c["nmu"], c["nt"], c["lmax"], c["precision"], c["batch"], c["grids"])
    if c["entry"] == "host":
        host = torch.empty(field.shape, dtype=field.dtype, pin_memory=True)
        host.copy_(field)
        out = torch.empty(plan.out_shape(c["batch"]), dtype=torch.float64, pin_memory=True)
        return {"case": c, "plan": plan, "keep": (host, out), "host": host.numpy(), "host_out": out.numpy()}
    s = {"case": c, "plan": plan, "field": field, "ws": plan.workspace(c["batch"]),
         "out": torch.empty(plan.out_shape(c["batch"]), dtype=torch.float64, device="cuda")}
    if c["entry"] == "graph":
        s["graph"] = plan.graph(field, s["ws"], s["out"])
    return s


def run(state):
    s = state
    c = s["case"]
    if c["entry"] == "shell":
        return [s["plan"].estimate(s["field"], s["ws"]).float()]
    if c["entry"] == "host":
        out = s["plan"].estimate_host(s["host"], out=s["host_out"])
        return list(out if c["precision"] == "fp64" else out.astype(np.float32))
    if c["entry"] == "graph":
        s["graph"].launch()
        out = s["out"]
    else:
        out = s["plan"].estimate(s["field"], s["ws"], out=s["out"])
    return list(out if c["precision"] == "fp64" else out.float())


# ------------------------------------------------------------------------------------------------
# The estimator's definitions in 64 bits, in plain numpy and torch (Gill & Bharadwaj, arXiv:2405.14513,
# Sec. II): rings in planes perpendicular to the line of sight, triple sums of ring fields, Y_lm weights
def _rings(ng):
    """Squared edges (times 9) of the rings, their mode-averaged radii, and the modes' 9 |u|^2."""
    e3 = [0]
    while e3[-1] < ng:
        e3.append(min(e3[-1] + (3 << ((len(e3) - 1) // 10)), ng))
    i = np.arange(-(ng // 2), ng // 2, dtype=np.int64)
    q = i[:, None] ** 2 + i[None, :] ** 2
    kperp = []
    for r in range(len(e3) - 1):
        m = (9 * q >= e3[r] ** 2) & (9 * q < e3[r + 1] ** 2)
        kperp.append(float(np.cumsum(np.sqrt(q[m].astype(np.float64)))[-1] / m.sum()))
    return e3, np.array(kperp)


def _masks(ng, e3, dims):
    f = torch.fft.fftfreq(ng, d=1.0 / ng, dtype=torch.float64, device=_device()).round().long()
    q = f[:, None] ** 2 + f[None, :] ** 2
    if dims == 3:
        q = q[:, :, None] + f[None, None, :] ** 2
    return [(9 * q >= a * a) & (9 * q < b * b) for a, b in zip(e3, e3[1:])], f, q


def _delta(field, box):
    ng = field.shape[0]
    d = torch.fft.fftn(field.double()) * (box ** 3 / ng ** 3)
    d[0, 0, 0] = 0.0
    return d


def _bin_half(x, n):
    edges = 0.5 + np.arange(1, n) / (2.0 * n)
    return np.searchsorted(edges, x, side="right")


def _shape(edges, kf, q1, q2, q3):
    """Acceptance, k1 bin, t, h = 1 - mu of triangles with squared sides q1, q2, q3."""
    ok = (q3 > 0) & (q2 >= q3) & (q1 >= q2)
    a1, a2, a3 = np.sqrt(q1), np.sqrt(q2), np.sqrt(q3)
    k = kf * a1
    ok &= (k >= edges[0]) & (k <= edges[-1])
    with np.errstate(invalid="ignore", divide="ignore"):
        t = a2 / a1
        h = np.clip((a3 - a1 + a2) * (a3 + a1 - a2) / (2.0 * a1 * a2), 0.0, 0.5)
    ok &= t >= 0.5
    ib = np.minimum(np.searchsorted(edges, k, side="right") - 1, len(edges) - 2)
    return ok, ib, t, h, a1, a2


def _legendre(lmax, x):
    """N_lm P_l^m(x) (orthonormal Y_lm without the azimuth, Condon-Shortley phase)."""
    P = {(0, 0): np.ones_like(x)}
    s = np.sqrt(np.maximum(0.0, 1.0 - x * x))
    for m in range(lmax + 1):
        if m:
            P[m, m] = -(2 * m - 1) * s * P[m - 1, m - 1]
        for l in range(m + 1, lmax + 1):
            P[l, m] = ((2 * l - 1) * x * P[l - 1, m] - ((l + m - 1) * P[l - 2, m] if l > m + 1 else 0.0)) / (l - m)
    return {(l, m): math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m)) * p
            for (l, m), p in P.items()}


def _exact_rings(c, seed, nfields):
    ng, box, lmax = c["ng"], c["box"], c["lmax"]
    dev, kf, nz, npts = _device(), 2.0 * math.pi / box, ng // 3, ng * ng
    edges = _edges(c)
    e3, kp = _rings(ng)
    nr = len(kp)
    masks, _, _ = _masks(ng, e3, 2)
    unit = torch.stack([torch.fft.fft2(m.double()).real.reshape(-1) for m in masks])         # [r][x]
    ntri = np.empty((nr, nr, nr))
    for r in range(nr):
        ntri[r] = ((unit * unit[r]) @ unit.T / npts).round().cpu().numpy()
    cubes = [_delta(field, box) for field in _fields(c, seed)[:nfields]]
    D = []                               # D[f][n] = [r][x] of plane n >= 0
    for cube in cubes:
        D.append([torch.stack([torch.fft.fft2(torch.where(m, cube[:, :, n], 0.0)).reshape(-1) for m in masks])
                  for n in range(nz + 1)])
    per_l = [int(g) for g in c["grids"].split(",")] if c["grids"] else None
    views = []
    for l in range(0, lmax + 1, 2):
        g = (per_l[l // 2],) * 2 if per_l else (c["nmu"], c["nt"])
        if views and views[-1][1] == g:
            views[-1][0].append(l)
        else:
            views.append(([l], g))
    lms = [[(l, m) for l in ls for m in range(l + 1)] for ls, _ in views]
    num = [np.zeros((nfields, c["nk1"] * g[0] * g[1], len(lm))) for (_, g), lm in zip(views, lms)]
    den = [np.zeros((c["nk1"] * g[0] * g[1], len(lm))) for (_, g), lm in zip(views, lms)]
    k2 = kp * kp
    for n1 in range(nz + 1):
        for n2 in range(0 if n1 == 0 else -nz, nz + 1):
            n3 = -(n1 + n2)
            if abs(n3) > nz:
                continue
            q1 = (k2 + float(n1) * n1)[:, None, None]
            q2 = (k2 + float(n2) * n2)[None, :, None]
            q3 = (k2 + float(n3) * n3)[None, None, :]
            q1, q2, q3 = np.broadcast_arrays(q1, q2, q3)
            ok, ib, t, h, a1, a2 = _shape(edges, kf, q1, q2, q3)
            ok &= ntri > 0
            if not ok.any():
                continue
            r1, r2, r3 = np.nonzero(ok)
            ib, t, h, a1, a2 = ib[ok], t[ok], h[ok], a1[ok], a2[ok]
            mu, nt, pz = 1.0 - h, ntri[ok], n1 / a1
            deg = mu >= 1.0 - 1e-12
            with np.errstate(invalid="ignore", divide="ignore"):
                px = ((a2 * mu - a1) * pz - n3) / (a2 * np.sqrt(h * (2.0 - h)))
                rho2 = 1.0 - pz * pz
                cphi = np.where(~deg & (rho2 > 0), np.clip(px / np.sqrt(np.maximum(rho2, 1e-300)), -1.0, 1.0), 1.0)
            rows, inv = np.unique(r1 * nr + r2, return_inverse=True)
            i1, i2 = torch.as_tensor(rows // nr, device=dev), torch.as_tensor(rows % nr, device=dev)
            sums = []
            for f in range(nfields):
                d1, d2, d3 = (D[f][abs(n)] if n >= 0 else D[f][-n].conj() for n in (n1, n2, n3))
                P, E = d1[i1] * d2[i2], d3
                sums.append((P.real @ E.real.T - P.imag @ E.imag.T))                          # Re sum_x D1 D2 D3
            S = torch.stack(sums)[:, torch.as_tensor(inv, device=dev), torch.as_tensor(r3, device=dev)].cpu().numpy()
            mult = 1.0 if n1 == 0 and n2 == 0 else 2.0
            Y = _legendre(lmax, pz)
            phi = np.arccos(cphi)
            for v, ((ls, g), lm) in enumerate(zip(views, lms)):
                b = (ib * g[0] + _bin_half(mu, g[0])) * g[1] + _bin_half(t, g[1])
                for j, (l, m) in enumerate(lm):
                    y = Y[l, m]
                    w = mult * (y if m == 0 else np.where(deg, 0.0, y * np.cos(m * phi)))
                    for f in range(nfields):
                        num[v][f, :, j] += np.bincount(b, weights=w * S[f], minlength=num[v].shape[1])
                    den[v][:, j] += np.bincount(b, weights=mult * y * y * nt, minlength=num[v].shape[1])
    out = []
    for f in range(nfields):
        blocks = []
        for v, ((ls, g), lm) in enumerate(zip(views, lms)):
            pref = np.array([math.sqrt((2 * l + 1) / (4 * math.pi)) for l, m in lm]) / (box ** 3 * npts)
            with np.errstate(invalid="ignore", divide="ignore"):
                B = np.where(den[v] > 0, pref * num[v][f] / den[v], np.nan)
            blocks.append(B.reshape(c["nk1"], g[0], g[1], len(lm)) if len(views) == 1 else B.reshape(-1))
        out.append(blocks[0] if len(views) == 1 else np.concatenate(blocks))
    return out


def _exact_shells(c, seed):
    ng, box, nl = c["ng"], c["box"], c["lmax"] // 2 + 1
    e3, _ = _rings(ng)
    ns = len(e3) - 1
    masks, f, q = _masks(ng, e3, 3)
    n3 = float(ng) ** 3
    K = []
    for m in masks:
        v = torch.sqrt(q[m].double())
        K.append(float(v.sum() / max(1, v.numel())))
    K = np.array(K)
    d = _delta(_fields(c, seed)[0], box)
    mu = (f[None, None, :] / torch.sqrt(q.clamp(min=1).double())).cpu().numpy()
    Y = _legendre(c["lmax"], mu)
    Y = [torch.as_tensor(Y[2 * i, 0], device=d.device) for i in range(nl)]

    def back(spec):
        return torch.fft.fftn(spec).real.reshape(-1)

    F = [[back(torch.where(m, d * y, 0.0)) for y in Y] for m in masks]                      # Delta Y_l0
    G = [back(torch.where(m, d, 0.0)) for m in masks]
    U = [back(m.double()) for m in masks]
    W = [[back(torch.where(m, y * y, 0.0)) for y in Y] for m in masks]
    edges, kf = _edges(c), 2.0 * math.pi / box
    num = np.zeros((c["nk1"] * c["nmu"] * c["nt"], nl))
    den = np.zeros_like(num)
    k2 = K * K
    for s1 in range(1, ns):
        for s2 in range(1, s1 + 1):
            s3 = np.arange(1, s2 + 1)
            ok, ib, t, h, _, _ = _shape(edges, kf, np.full(s2, k2[s1]), np.full(s2, k2[s2]), k2[s3])
            for k in np.flatnonzero(ok):
                UU, GG = U[s2] * U[s3[k]], G[s2] * G[s3[k]]
                if round(float(U[s1] @ UU) / n3) < 1:
                    continue
                b = (ib[k] * c["nmu"] + _bin_half(1.0 - h[k], c["nmu"])) * c["nt"] + _bin_half(t[k], c["nt"])
                for i in range(nl):
                    num[b, i] += float(F[s1][i] @ GG) / n3
                    den[b, i] += float(W[s1][i] @ UU) / n3
    pref = np.sqrt((4 * np.arange(nl) + 1) / (4 * math.pi)) / box ** 3
    with np.errstate(invalid="ignore", divide="ignore"):
        B = np.where(den > 0, pref * num / den, np.nan)
    return [B.reshape(c["nk1"], c["nmu"], c["nt"], nl)]


def exact(case, seed):
    c = case
    if c["entry"] == "shell":
        return _exact_shells(c, seed)
    # the sums below take about ng^7.3: a second or two a field at 128^3, minutes at 256^3
    if c["ng"] > 128:
        return None
    n = min(c["batch"], {128: 3, 96: 6}.get(c["ng"], 16))
    return _exact_rings(c, seed, n) + [None] * (c["batch"] - n)


# ------------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _sums(ng, lo, hi):
    """Grid points of all triple sums and of all distinct pair products D1 D2, each on the smallest
    reduction grid (F x 2^q, F = 1, 3, 5, 7) on which its sum is exact, k1 between lo and hi (grid units)."""
    e3, kp = _rings(ng)
    dev = _device()
    nz = ng // 3
    e = torch.tensor(e3, dtype=torch.float64, device=dev) / 3
    maxc = torch.ceil(e[1:]) - 1
    grids = torch.tensor(sorted({f * 2 ** q for f in (1, 3, 5, 7) for q in range(2, 11) if 8 <= f * 2 ** q <= ng}),
                         dtype=torch.float64, device=dev)
    need = (maxc[:, None, None] + maxc[None, :, None] + maxc[None, None, :] + 1).clamp(max=float(ng))
    lev = torch.searchsorted(grids, need)
    m2 = grids[lev] ** 2
    a, b = e[:-1], e[1:]
    tri = (a[:, None, None] < b[None, :, None] + b[None, None, :]) & (a[None, :, None] < b[:, None, None] + b[None, None, :]) \
        & (a[None, None, :] < b[:, None, None] + b[None, :, None])
    k2 = torch.as_tensor(kp ** 2, device=dev)
    triple = pair = 0.0
    for n1 in range(nz + 1):
        n2 = torch.arange(0 if n1 == 0 else -nz, nz - n1 + 1, dtype=torch.float64, device=dev)[:, None, None, None]
        q1, q2 = (k2 + n1 * n1)[None, :, None, None], k2[None, None, :, None] + n2 * n2
        q3 = k2[None, None, None, :] + (n1 + n2) ** 2
        ok = tri & (q1 >= q2) & (q2 >= q3) & (q3 > 0) & (q2 >= 0.25 * q1) & (q1 >= lo * lo) & (q1 <= hi * hi)
        triple += float((ok.sum(0) * m2).sum())
        for g in range(len(grids)):
            pair += float((ok & (lev == g)).any(3).sum()) * float(grids[g]) ** 2
    return triple, pair


def work(case):
    c = case
    ng, n3 = c["ng"], float(c["ng"]) ** 3
    item = 8 if c["precision"] == "fp64" else 4
    fft = 2.5 * n3 * math.log2(n3)
    if c["entry"] == "shell":
        e3, _ = _rings(ng)
        nl, ns = c["lmax"] // 2 + 1, len(e3) - 2
        triples = ns * (ns + 1) * (ns + 2) / 6 * 0.4
        return {"bytes": n3 * 4 + 8.0 * c["nk1"] * c["nmu"] * c["nt"] * nl, "flops": fft * (1 + ns * nl) + 3.0 * n3 * nl * triples}
    triple, pair = _sums(ng, c["lo"] * ng, c["hi"] * ng)
    per_l = [int(g) ** 2 for g in c["grids"].split(",")] if c["grids"] else [c["nmu"] * c["nt"]] * (c["lmax"] // 2 + 1)
    outs = c["nk1"] * sum(g * (2 * i + 1) for i, g in enumerate(per_l))
    return {"bytes": c["batch"] * (n3 * item + 8.0 * outs), "flops": c["batch"] * (fft + 4.0 * triple + 6.0 * pair)}
