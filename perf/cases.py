"""What this framework's users have it do: twelve calls through its public entry points, over the real range of sizes.

Each case is one call (or the few calls that always go together) of map-making: the normal operator
P^T N^-1 P in its precisions and pointing modes, the right-hand side, the set-up of a solve, whole
solves, the simulation and binning of data, chi^2 with its gradients, and gap filling. Scans are the
spinning, precessing satellite the benchmarks use (20 Hz, spin 1 rpm at 50 degrees, precession 1 h at
45 degrees), focal planes are hexagonal of radius 5 degrees, the noise is 1/f + white with a 64-tap
banded inverse, the sky Gaussian. The seed sets the start of the scan, the sky, the noise levels of
the detectors, the noise and the gaps.

``exact`` restates each call in FP64 with plain torch (its own pointing, band, sums and conjugate
gradients); integer and boolean outputs have no value there.
"""
import math
import random

import numpy as np
import torch

import paper_2603_19600_gb300 as fx

FSAMP, SIGMA, FKNEE = 20.0, 10.0, 0.1
EPOCH = 10 ** 6           # scans start within this many seconds of the epoch
CHUNK = 1 << 24           # samples handled at once where inputs and exact values are made
F64 = torch.float64


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


# ------------------------------------------------------------------------------------------ cases
def _case(kind, ndet, nsamp, nside, **kw):
    c = dict(kind=kind, ndet=ndet, nsamp=nsamp, nside=nside, nobs=1, mode="cache_f32", precision="f32", acc="f64",
             ntaps=64, white=False)
    c.update(kw)
    return c


def listed():
    cases = {
        # the smallest whole call: four detectors on a coarse map, plain FP64, white noise;
        # launches and host work count
        "solve_small_white_f64": _case("solve", 4, 65536, 16, mode="cache_f64", precision="f64", white=True),
        # a whole mixed-precision solve to a true residual of 1e-8 (FP32 inner, FP64-accurate outer)
        "solve_mixed": _case("solve", 64, 131072, 256, mode="cache_mixed"),
        # the inner operator of a solve at full size: cached FP32 pointing, FP64 per-pixel sums
        "normal_f32_full": _case("normal", 256, 1 << 20, 512),
        # the same on a ragged batch of three short observations with compensated FP32 sums
        "normal_f32_ragged_kahan": _case("normal", 24, 66537, 128, nobs=3, acc="f32_kahan"),
        # the operator of a plain FP64 solve on a medium observation
        "normal_f64": _case("normal", 32, 262147, 256, mode="cache_f64", precision="f64"),
        # pointing too large to keep: recomputed from the quaternions in every application
        "normal_on_the_fly": _case("normal", 64, 1 << 18, 512, mode="on_the_fly"),
        # strongly correlated noise: a 1024-tap band, applied by overlap-save
        "normal_long_band": _case("normal", 64, 1 << 18, 512, ntaps=1024),
        # the right-hand side of a mixed solve, from FP32 data
        "rhs": _case("rhs", 128, 1 << 19, 512, mode="cache_mixed"),
        # what each solve begins with: pointing expanded from new quaternions, block-Jacobi blocks
        "setup": _case("setup", 96, 300007, 512),
        # simulation: a sky observed into time-ordered data and binned back with its hit counts
        "simulate_and_bin": _case("simulate", 48, 262143, 256),
        # one step of fitting map and polarisation angles: chi^2 and both gradients through autograd
        "chi2_grad": _case("chi2", 128, 1 << 17, 256, mode="cache_f64", precision="f64"),
        # glitches cut from the data filled by a constrained realisation of the noise
        "gapfill": _case("gapfill", 32, 131071, 256, precision="f64"),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "normal", "normal", "normal", "rhs", "setup", "simulate", "chi2", "gapfill"])
    top = {"normal": 256 << 20, "rhs": 64 << 20, "setup": 32 << 20, "simulate": 32 << 20, "solve": 8 << 20,
           "chi2": 16 << 20, "gapfill": 4 << 20}[kind]
    nside = rng.choice([16, 32, 64, 128, 256, 512])
    total = _log(rng, 4 * 65536, top)
    ndet = min(256, max(1, _log(rng, 4, 256)))
    nsamp = min(1 << 20, max(4097, total // ndet))
    ndet = max(1, min(256, total // nsamp))
    if kind == "normal":
        mode, precision = rng.choice([("cache_f32", "f32"), ("cache_f32", "f32"), ("cache_f64", "f64"),
                                      ("cache_mixed", "f32x2"), ("on_the_fly", "f32")])
        acc, ntaps, nobs = rng.choice(["f64", "f64", "f32_kahan"]), rng.choice([64, 64, 33, 1024]), rng.choice([1, 1, 2, 5])
        if (mode, acc) != ("cache_f32", "f64") or ntaps > 64 or nobs > 1:   # these cost more per sample
            ndet = max(1, min(ndet, (16 << 20) // nsamp))
        return _case(kind, ndet, nsamp, nside, mode=mode, precision=precision, nobs=nobs, acc=acc, ntaps=ntaps)
    if kind == "solve":
        nside = max(n for n in (16, 32, 64, 128, 256) if n == 16 or (n <= nside and 48 * n * n <= ndet * nsamp))
        mode, precision = rng.choice([("cache_f64", "f64"), ("cache_mixed", "f32")])
        return _case(kind, max(4, ndet), nsamp, nside, mode=mode, precision=precision, white=rng.random() < 0.3)
    if kind == "rhs":
        return _case(kind, ndet, nsamp, nside, mode=rng.choice(["cache_f32", "cache_mixed"]))
    if kind == "chi2":
        return _case(kind, ndet, nsamp, nside, mode="cache_f64", precision=rng.choice(["f64", "f32x2"]))
    if kind == "gapfill":
        return _case(kind, ndet, nsamp, nside, precision=rng.choice(["f64", "f32x2"]))
    return _case(kind, ndet, nsamp, nside)


def _shapes(case):
    """(ndet, nsamp, nside) per observation: the later ones of a batch are smaller and coarser."""
    nd, ns, n = case["ndet"], case["nsamp"], case["nside"]
    return [(max(1, nd - i * (nd // 6)), ns - i * (ns // 8) - i, n if i % 2 == 0 else max(1, n // 2))
            for i in range(case["nobs"])]


# ----------------------------------------------------------------------------------------- inputs
def _qmul(a, b):
    aw, ax, ay, az = a.unbind(-1)
    bw, bx, by, bz = b.unbind(-1)
    return torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                        aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], -1)


def _rot(axis, angle):
    angle = torch.as_tensor(angle, dtype=F64, device=_dev())
    q = torch.zeros(angle.shape + (4,), dtype=F64, device=angle.device)
    q[..., 0] = torch.cos(angle / 2)
    q[..., axis + 1] = torch.sin(angle / 2)
    return q


def _scan(nsamp, t0):
    """Boresight quaternions (w, x, y, z) of the satellite scan from time t0 (seconds)."""
    t = t0 + torch.arange(nsamp, dtype=F64, device=_dev()) / FSAMP
    q = _rot(2, 2 * math.pi / (365.25 * 86400.0) * t)
    for axis, angle in ((1, math.pi / 2), (2, 2 * math.pi / 3600.0 * t), (1, math.radians(45.0)),
                        (2, 2 * math.pi / 60.0 * t), (1, math.radians(50.0))):
        q = _qmul(q, _rot(axis, angle).expand_as(q))
    return q / torch.linalg.vector_norm(q, dim=-1, keepdim=True)


def _focal_plane(ndet):
    """Detector quaternions of the ndet lattice points nearest the centre of a hexagonal plane."""
    k = int(math.ceil(math.sqrt(ndet))) + 2
    pts = sorted((m * m + m * n + n * n, math.atan2(n * math.sqrt(3.0) / 2, m + n / 2) % (2 * math.pi))
                 for m in range(-k, k + 1) for n in range(-k, k + 1))[:ndet]
    rad = np.sqrt(np.array([p[0] for p in pts], float))
    rad = math.radians(5.0) * (rad / rad.max() if rad.max() > 0 else rad)
    ang = torch.as_tensor([p[1] for p in pts], dtype=F64, device=_dev())
    psi = math.radians(45.0) * (torch.arange(ndet, device=_dev()) % 4)
    q = _qmul(_rot(2, ang), _rot(1, torch.as_tensor(rad, device=_dev())))
    q = _qmul(q, _qmul(_rot(2, -ang), _rot(2, psi)))
    return q / torch.linalg.vector_norm(q, dim=-1, keepdim=True)


def _psd_taps(ntaps, inverse):
    """Band c_0 .. c_{ntaps-1} of the (inverse) covariance of 1/f + white noise, Bartlett-tapered."""
    f = np.fft.rfftfreq(1 << 16, d=1.0 / FSAMP)
    if inverse:
        psd = np.zeros_like(f)
        psd[1:] = 1.0 / (SIGMA ** 2 * (1.0 + FKNEE / f[1:]))
    else:
        psd = SIGMA ** 2 * (1.0 + FKNEE / np.sqrt(f ** 2 + 0.01 ** 2))
    return np.fft.irfft(psd)[:ntaps] * (1.0 - np.arange(ntaps) / ntaps)


def _noise(g, ndet, nsamp, dtype):
    """1/f + white noise [ndet][nsamp], shaped in Fourier space."""
    n = 1 << max(12, (nsamp - 1).bit_length())
    f = torch.fft.rfftfreq(n, d=1.0 / FSAMP, device=_dev(), dtype=torch.float32)
    amp = SIGMA * torch.sqrt(1.0 + FKNEE / f.clamp_min(float(f[1])))
    amp[0] = 0.0
    out = torch.empty(ndet, nsamp, dtype=dtype, device=_dev())
    step = max(1, CHUNK // n)
    for a in range(0, ndet, step):
        w = torch.randn(min(step, ndet - a), n, generator=g, device=_dev())
        out[a:a + step] = torch.fft.irfft(torch.fft.rfft(w) * amp, n=n)[:, :nsamp].to(dtype)
    return out


class _Inputs:
    """The arrays a user's program starts from, made from the seed alone."""

    def __init__(self, case, seed):
        self.case, self.shapes = case, _shapes(case)
        g = self.g = torch.Generator(device=_dev()).manual_seed(seed)
        t0 = random.Random(seed).uniform(0.0, EPOCH)
        self.q_bore = [_scan(ns, t0 + 1e5 * i) for i, (_, ns, _) in enumerate(self.shapes)]
        self.q_det = [_focal_plane(nd) for nd, _, _ in self.shapes]
        self.npix = [12 * n * n for _, _, n in self.shapes]
        nd = sum(s[0] for s in self.shapes)
        level = torch.exp(0.1 * torch.randn(nd, 1, generator=g, device=_dev(), dtype=F64))   # noise levels
        if case["white"]:
            self.params = level.reshape(-1) * SIGMA ** 2
        else:
            taps = torch.as_tensor(_psd_taps(case["ntaps"], case["kind"] != "gapfill"), device=_dev())
            self.params = (level if case["kind"] == "gapfill" else 1.0 / level) * taps
        self.psi = None
        if case["kind"] == "chi2":
            self.psi = math.radians(1.0) * torch.randn(nd, generator=g, device=_dev(), dtype=F64)
        self.sky = torch.randn(sum(self.npix), 3, generator=g, device=_dev(), dtype=F64)
        self.sky *= torch.tensor([100.0, 1.0, 1.0], device=_dev(), dtype=F64)

    def tod(self, dtype):
        """d = P sky + noise, flat over observations."""
        parts, p0 = [], 0
        for i, (nd, ns, _) in enumerate(self.shapes):
            d = _noise(self.g, nd, ns, dtype)
            for a, b, pix, c, s in self.pointing(i):
                d[a:b] += _project(self.sky[p0:p0 + self.npix[i]], pix, c, s).to(dtype)
            parts.append(d.reshape(-1))
            p0 += self.npix[i]
        return torch.cat(parts)

    def gaps(self):
        """Data, gap mask (single samples and stretches of 120) and noise realisation of gap filling."""
        (nd, ns, _), case = self.shapes[0], self.case
        hit = torch.rand(nd, ns, generator=self.g, device=_dev()) < 0.05
        starts = (torch.rand(nd, ns, generator=self.g, device=_dev()) < 3e-4).to(torch.int32).cumsum(1)
        long_gap = starts.clone()
        long_gap[:, 120:] -= starts[:, :-120]
        valid = ~(hit | (long_gap > 0))
        n = 1 << (ns + 2 * case["ntaps"]).bit_length()
        kern = torch.zeros(nd, n, dtype=F64, device=_dev())
        kern[:, :case["ntaps"]] = self.params
        kern[:, n - case["ntaps"] + 1:] = self.params[:, 1:].flip(1)
        amp = torch.fft.rfft(kern).real.clamp_min(0.0).sqrt()
        w = torch.randn(2, nd, n, generator=self.g, device=_dev(), dtype=F64)
        d, nr = torch.fft.irfft(torch.fft.rfft(w) * amp, n=n)[:, :, :ns].to(torch.float32)
        return (d + 2.0).reshape(-1), valid.to(torch.uint8).reshape(-1), nr.reshape(-1).contiguous()

    def pointing(self, i, psi=None):
        """Pixel and weights of observation i in FP64, a block of detectors at a time."""
        nd, ns, nside = self.shapes[i]
        step = max(1, CHUNK // ns)
        for a in range(0, nd, step):
            pix, c, s = _point(self.q_bore[i], self.q_det[i][a:a + step], nside)
            if psi is not None:
                c2, s2 = torch.cos(2 * psi[a:a + step, None]), torch.sin(2 * psi[a:a + step, None])
                c, s = c * c2 - s * s2, s * c2 + c * s2
            yield a, a + pix.shape[0], pix, c, s


def _axes(q, col):
    w, x, y, z = q.unbind(-1)
    if col == 0:
        return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y)], -1)
    if col == 1:
        return torch.stack([2 * (x * y - w * z), 1 - 2 * (x * x + z * z), 2 * (y * z + w * x)], -1)
    return torch.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)], -1)


def _point(qb, qd, nside):
    """HEALPix RING pixel and (cos 2 psi, sin 2 psi) of every detector and sample, in FP64."""
    cols = [_axes(qb, k) for k in range(3)]
    los, ori = _axes(qd, 2), _axes(qd, 0)

    def turn(v, r):
        return v[:, 0:1] * cols[0][:, r] + v[:, 1:2] * cols[1][:, r] + v[:, 2:3] * cols[2][:, r]

    dx, dy, dz = (turn(los, r) for r in range(3))
    ox, oy, oz = (turn(ori, r) for r in range(3))
    rho2 = dx * dx + dy * dy
    a = rho2 * oz - dz * (ox * dx + oy * dy)
    b = oy * dx - ox * dy
    n2 = (a * a + b * b).clamp_min(1e-300)
    c, s = (a * a - b * b) / n2, 2 * a * b / n2
    tt = (torch.atan2(dy, dx) * (2 / math.pi)) % 4.0
    za = dz.abs()
    t1, t2 = nside * (0.5 + tt), nside * 0.75 * dz
    jp, jm = torch.floor(t1 - t2).long(), torch.floor(t1 + t2).long()
    ir = nside + 1 + jp - jm
    ip = torch.div(jp + jm - nside + 1 - (ir & 1), 2, rounding_mode="floor") % (4 * nside)
    belt = 2 * nside * (nside - 1) + (ir - 1) * 4 * nside + ip
    tp = tt - torch.floor(tt)
    tmp = nside * torch.sqrt(3 * rho2 / (1 + za))
    ir = torch.floor(tp * tmp).long() + torch.floor((1 - tp) * tmp).long() + 1
    ip = torch.floor(tt * ir).long() % (4 * ir)
    cap = torch.where(dz > 0, 2 * ir * (ir - 1) + ip, 12 * nside * nside - 2 * ir * (ir + 1) + ip)
    return torch.where(za <= 2.0 / 3.0, belt, cap), c, s


def _project(m, pix, c, s):
    v = m[pix]
    return v[..., 0] + v[..., 1] * c + v[..., 2] * s


def prepare(case, seed):
    inp = _Inputs(case, seed)
    nd, ns, nside = ([s[k] for s in inp.shapes] for k in range(3))
    st = {"case": case, "P": fx.Pointing(torch.cat(inp.q_bore), torch.cat(inp.q_det), nd, ns, nside, psi_offset=inp.psi,
                                         mode=case["mode"])}
    st["N"] = (fx.Noise.white if case["white"] else fx.Noise.banded)(st["P"], inp.params)
    kind = case["kind"]
    if kind == "solve":
        st["d"] = inp.tod(F64 if case["precision"] == "f64" else torch.float32)
        st["stream"] = torch.cuda.Stream()
    elif kind in ("normal", "simulate"):
        st["x"] = inp.sky
    elif kind == "rhs":
        st["d"] = inp.tod(torch.float32)
    elif kind == "chi2":
        st["d"] = inp.tod(F64)
        st["m"] = (1.01 * inp.sky).requires_grad_(True)
        st["psi"] = (0.5 * inp.psi).requires_grad_(True)
    elif kind == "gapfill":
        st["d"], st["valid"], st["n_real"] = inp.gaps()
    torch.cuda.synchronize()
    return st


# -------------------------------------------------------------------------------------------- run
def run(st):
    case, P, N = st["case"], st["P"], st["N"]
    kind = case["kind"]
    if kind == "normal":
        return fx.ptnp_apply(P, N, st["x"], precision=case["precision"], acc=case["acc"])
    if kind == "rhs":
        return fx.rhs(P, N, st["d"])
    if kind == "setup":
        P.refresh()
        b = fx.blockdiag_precond(P, N)
        pix, c, s = P.cache()
        return {"pix": pix, "c": c, "s": s, "inv": b["inv"], "valid": b["valid"], "hits": b["hits"], "rcond": b["rcond"]}
    if kind == "simulate":
        tod = P.apply(st["x"], dtype=torch.float32)
        m, hits = P.transpose(tod, hits=True)
        return {"tod": tod, "map": m, "hits": hits}
    if kind == "chi2":
        v = fx.chi2(st["m"], st["psi"], P, N, st["d"], case["precision"])
        gm, gp = torch.autograd.grad(v, (st["m"], st["psi"]))
        return {"chi2": v.detach(), "grad_map": gm, "grad_psi": gp}
    if kind == "gapfill":
        out, _, _ = fx.gapfill(N, st["d"], st["valid"], st["n_real"], precision=case["precision"])
        return out
    if case["precision"] == "f64":
        x, valid, _ = fx.mapmaker_cg(P, N, st["d"], maxiter=60, tol=1e-12)
        return {"map": x, "valid": valid}
    # as a pipeline does: the solve on a stream of its own, its iterations as a CUDA graph
    with torch.cuda.stream(st["stream"]):
        x, valid, _ = fx.mapmaker_cg(P, N, st["d"], maxiter=100, tol=1e-8, precision="f32", acc=case["acc"])
        return {"map": x, "valid": valid}


def work(case):
    shapes = _shapes(case)
    n = sum(a * b for a, b, _ in shapes)
    bore = 32 * sum(b for _, b, _ in shapes)
    npix = sum(12 * k * k for _, _, k in shapes)
    per = {"on_the_fly": 0, "cache_f32": 12, "cache_f64": 20, "cache_mixed": 20}[case["mode"]]
    if case["precision"] == "f32" and case["kind"] == "normal":
        per = min(per, 12)
    otf = bore if case["mode"] == "on_the_fly" else 0
    band = 2 if case["white"] else 2 * (2 * case["ntaps"] - 1)
    if case["ntaps"] > 64:   # by transforms of 8192 points
        band = 2 * 5 * 13
    kind = case["kind"]
    if kind == "normal":
        return {"bytes": per * n + otf + 48 * npix, "flops": n * (band + 10)}
    if kind == "rhs":
        return {"bytes": (per + 4) * n + 24 * npix, "flops": n * (band + 6)}
    if kind == "setup":
        return {"bytes": bore + 12 * n + 12 * n + 24 * n + (48 + 8 + 1 + 4) * npix, "flops": n * 120}
    if kind == "simulate":
        return {"bytes": 2 * per * n + 8 * n + (24 + 24 + 4) * npix, "flops": n * 10}
    if kind == "chi2":
        return {"bytes": (per + 8) * n + 48 * npix, "flops": n * (band + 20)}
    if kind == "gapfill":   # data, mask, realisation, result; some 30 band products
        return {"bytes": (4 + 1 + 4 + 4) * n, "flops": n * 30 * (band + 12)}
    iters = 2 if case["white"] else 16   # right-hand side, preconditioner, iterations, residual
    size = 8 if case["precision"] == "f64" else 4
    return {"bytes": (size + per * (iters + 3)) * n + 200 * npix * iters, "flops": n * (iters + 2) * (band + 10)}


# ------------------------------------------------------------------------------------------ exact
def _band(x, taps):
    """Symmetric band along each row: y_t = sum_{|k| < K} c_|k| x_{t+k}, zeros outside the row."""
    k, ns = taps.shape[1], x.shape[1]
    if k > 64:
        n = 1 << (ns + 2 * k).bit_length()
        kern = torch.zeros(x.shape[0], n, dtype=F64, device=x.device)
        kern[:, :k] = taps
        kern[:, n - k + 1:] = taps[:, 1:].flip(1)
        return torch.fft.irfft(torch.fft.rfft(x, n=n) * torch.fft.rfft(kern).real, n=n)[:, :ns]
    y = taps[:, 0:1] * x
    for j in range(1, min(k, ns)):
        y[:, j:] += taps[:, j:j + 1] * x[:, :-j]
        y[:, :-j] += taps[:, j:j + 1] * x[:, j:]
    return y


def _weigh(inp, x, rows):
    p = inp.params[rows]
    return x / p[:, None] if inp.case["white"] else _band(x, p)


def _scatter(out, y, pix, c, s):
    pix = pix.reshape(-1)
    for k, v in enumerate((y, y * c, y * s)):
        out[:, k].index_add_(0, pix, v.reshape(-1))


def _sweep(inp, make, psi=None, each=None):
    """P^T N^-1 of make(obs, rows a:b, pix, c, s) over all observations."""
    outs, d0, p0 = [], 0, 0
    for i, (nd, _, _) in enumerate(inp.shapes):
        out = torch.zeros(inp.npix[i], 3, dtype=F64, device=_dev())
        ps = None if psi is None else psi[d0:d0 + nd]
        for a, b, pix, c, s in inp.pointing(i, ps):
            x = make(i, a, b, p0, pix, c, s)
            y = _weigh(inp, x, slice(d0 + a, d0 + b))
            _scatter(out, y, pix, c, s)
            if each is not None:
                each(d0 + a, d0 + b, p0, x, y, pix, c, s)
        outs.append(out)
        d0 += nd
        p0 += inp.npix[i]
    return torch.cat(outs)


def _normal(inp, m):
    return _sweep(inp, lambda i, a, b, p0, pix, c, s: _project(m[p0:p0 + inp.npix[i]], pix, c, s))


def _rhs(inp, d):
    def rows(i, a, b, p0, pix, c, s):
        o = sum(x * y for x, y, _ in inp.shapes[:i])
        ns = inp.shapes[i][1]
        return d[o + a * ns:o + b * ns].view(b - a, ns).to(F64)
    return _sweep(inp, rows)


def _blocks(inp):
    """Inverse 3x3 blocks of P^T diag(N^-1) P in full, their mask and reciprocal condition numbers."""
    (nd, _, _), npix = inp.shapes[0], inp.npix[0]
    m = torch.zeros(npix, 6, dtype=F64, device=_dev())
    hits = torch.zeros(npix, dtype=torch.int64, device=_dev())
    for a, b, pix, c, s in inp.pointing(0):
        w = (1.0 / inp.params[a:b, None] if inp.case["white"] else inp.params[a:b, 0:1]).expand_as(c)
        p = pix.reshape(-1)
        for k, v in enumerate((w, w * c, w * s, w * c * c, w * c * s, w * s * s)):
            m[:, k].index_add_(0, p, v.reshape(-1))
        hits.index_add_(0, p, torch.ones_like(p))
    full = m[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].view(npix, 3, 3)
    low, info = torch.linalg.cholesky_ex(full)
    ok = (hits >= 3) & (info == 0)
    eye = torch.eye(3, dtype=F64, device=_dev())
    inv = torch.cholesky_inverse(torch.where(ok[:, None, None], low, eye))
    norm1 = lambda x: x.abs().sum(1).amax(1)  # noqa: E731
    rcond = torch.where(ok, 1.0 / (norm1(full) * norm1(inv)), torch.zeros((), dtype=F64, device=_dev()))
    valid = ok & (rcond >= 1e-3)
    return torch.where(valid[:, None, None], inv, torch.zeros_like(inv)), valid, rcond


def _solve(inp, d):
    inv, valid, _ = _blocks(inp)
    pre = lambda r: torch.einsum("pij,pj->pi", inv, r)  # noqa: E731
    r = _rhs(inp, d) * valid[:, None]
    x, z = torch.zeros_like(r), pre(r)
    p, rz, bb = z.clone(), (r * z).sum(), (r * r).sum()
    for _ in range(60):
        q = _normal(inp, p) * valid[:, None]
        alpha = rz / (p * q).sum()
        x += alpha * p
        r -= alpha * q
        if float((r * r).sum() / bb) < 1e-28:
            break
        z = pre(r)
        rz, old = (r * z).sum(), rz
        p = z + (rz / old) * p
    return {"map": x, "valid": None}


def _fill(inp, d, valid, nr):
    nd, ns, _ = inp.shapes[0]
    v, d, nr = valid.view(nd, ns).bool(), d.view(nd, ns).to(F64), nr.view(nd, ns).to(F64)
    r = torch.where(v, d - nr, torch.zeros_like(d))
    y, p, rr = torch.zeros_like(r), r.clone(), (r * r).sum(1, keepdim=True)
    first = rr.clone()
    for _ in range(200):
        q = _band(p, inp.params) * v
        alpha = rr / (p * q).sum(1, keepdim=True).clamp_min(1e-300)
        y += alpha * p
        r -= alpha * q
        new = (r * r).sum(1, keepdim=True)
        if float((new / first.clamp_min(1e-300)).max()) < 1e-26:
            break
        p = r + (new / rr.clamp_min(1e-300)) * p
        rr = new
    return torch.where(v, d, nr + _band(y, inp.params)).reshape(-1)


def exact(case, seed):
    inp = _Inputs(case, seed)
    kind = case["kind"]
    if kind == "normal":
        return _normal(inp, inp.sky)
    if kind == "rhs":
        return _rhs(inp, inp.tod(torch.float32))
    if kind == "solve":
        return _solve(inp, inp.tod(F64 if case["precision"] == "f64" else torch.float32))
    if kind == "gapfill":
        return _fill(inp, *inp.gaps())
    if kind == "setup":
        inv, _, rcond = _blocks(inp)
        cs = [(c.reshape(-1), s.reshape(-1)) for _, _, _, c, s in inp.pointing(0)]
        return {"pix": None, "c": torch.cat([c for c, _ in cs]), "s": torch.cat([s for _, s in cs]),
                "inv": torch.stack([inv[:, 0, 0], inv[:, 0, 1], inv[:, 0, 2], inv[:, 1, 1], inv[:, 1, 2], inv[:, 2, 2]], 1),
                "valid": None, "hits": None, "rcond": rcond}
    if kind == "simulate":
        tod, out = [], torch.zeros(inp.npix[0], 3, dtype=F64, device=_dev())
        for _, _, pix, c, s in inp.pointing(0):
            v = _project(inp.sky, pix, c, s)
            _scatter(out, v, pix, c, s)
            tod.append(v.reshape(-1))
        return {"tod": torch.cat(tod), "map": out, "hits": None}
    d, m, psi = inp.tod(F64), 1.01 * inp.sky, 0.5 * inp.psi
    (_, ns, _), val, gp = inp.shapes[0], [], torch.zeros_like(psi)

    def each(a, b, p0, r, y, pix, c, s):
        val.append((r * y).sum())
        v = m[pix]
        gp[a:b] = -4.0 * (y * (v[..., 2] * c - v[..., 1] * s)).sum(1)

    gm = _sweep(inp, lambda i, a, b, p0, pix, c, s: d[a * ns:b * ns].view(b - a, ns) - _project(m, pix, c, s), psi, each)
    return {"chi2": torch.stack(val).sum(), "grad_map": -2.0 * gm, "grad_psi": gp}
