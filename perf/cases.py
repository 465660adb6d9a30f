"""Performance cases of the lensing remap: the work a user has this library do, through its public entry points.

Every case is one of four uses:

* ``lens``: ``Plan.lens`` on a contiguous RING range (or the whole sky) of one map, K nearest pixels per target;
* ``batch``: ``Batch.run`` over ranges of several resident maps of different Nside, K and spin;
* ``paper``: ``PaperPlan.lens`` / ``supersample``, the pixel-centred stencil with tabulated inverses;
* ``synth``: ``Synth.run``, harmonic synthesis of an unlensed map.

Maps are realisations of the field the estimator assumes (random plane waves whose wavenumbers follow the
spectrum, evaluated at the pixel centres; Q/U and vector fields are the wave's E-type derivatives), deflections
are gradients of such a potential with an rms of 2.5 arcmin, so that values and conditioning are those of a CMB
map being lensed.  ``exact`` recomputes a case in plain FP64 torch, with the correlation function summed directly.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1003_4984_gb300 as fl

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
NUGGET = 1.49e-8
DEFL_RMS = 2.5 * math.pi / (180.0 * 60.0)
WAVES = 24  # plane waves per field


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # a serving request below the loop's smallest chunk: one call's latency, a handful of warps
        _lens("lens_T_1009", 512, 0, 16, "mixed", 1009),
        # the whole small sky of the library's first configuration, FP64, with the error bars
        _lens("lens_T_sky64_fp64", 64, 0, 16, "fp64", 12 * 64 * 64, lmax=128, damp=100.0, variance=True),
        # an ordinary serving request (the job stream starts at 1e4 points), ragged
        _lens("lens_QU_20011", 1024, 2, 32, "mixed", 20011),
        # temperature at survey resolution, both precisions
        _lens("lens_T_2048", 2048, 0, 32, "mixed", 2097169, damp=2500.0),
        _lens("lens_T_2048_fp64", 2048, 0, 32, "fp64", 1048583, damp=2500.0),
        # polarisation at the largest resolution, a window of the resident sky, both precisions
        _lens("lens_QU_4096", 4096, 2, 32, "mixed", 4194304, damp=2500.0),
        _lens("lens_QU_4096_fp64", 4096, 2, 32, "fp64", 524309, damp=2500.0),
        # the widely linear estimator (xi+ and xi-)
        _lens("lens_QU_aug", 2048, 2, 32, "mixed", 262147, damp=2500.0, augmented=True),
        # many maps in one launch
        {"name": "batch_8", "use": "batch", "jobs": 8, "pick": 11, "points": 60000},
        # the paper's stencil: a whole temperature sky at y = 1, Q/U at y = 2 in FP64
        _paper("paper_T_y1", 2048, 0, 1, "mixed", 12 * 2048 * 2048),
        _paper("paper_QU_y2_fp64", 1024, 2, 2, "fp64", 2097169),
        # the unlensed Q/U map itself
        {"name": "synth_QU", "use": "synth", "nside": 1024, "lmax": 2048, "spin": 2, "precision": "mixed"},
    ]


def _lens(name, nside, spin, K, precision, count, lmax=None, damp=None, augmented=False, first=None, variance=False):
    # variance: a lensed map is made without it (the entry point's default); the small stencil asks for it, while with
    # 24 and more pixels of these band-limited fields it is 1e-6 of xi(0) down to the nugget's own share
    lmax = min(2 * nside, 4096) if lmax is None else lmax
    npix = 12 * nside * nside
    # by default a window that starts in the northern cap and, when long enough, crosses into the belt
    first = (npix - count) // 7 if first is None else first
    return {"name": name, "use": "lens", "nside": nside, "lmax": lmax, "damp": 0.61 * lmax if damp is None else damp,
            "spin": spin, "K": K, "precision": precision, "augmented": augmented, "variance": variance,
            "first": first, "count": count}


def _paper(name, nside, spin, y, precision, count, supersample=False, first=None):
    lmax = min(2 * nside, 4096)
    npix = 12 * nside * nside * (4 if supersample else 1)
    return {"name": name, "use": "paper", "nside": nside, "lmax": lmax, "damp": 0.61 * lmax, "spin": spin, "y": y,
            "precision": precision, "supersample": supersample,
            "first": (npix - count) // 7 if first is None else first, "count": count}


def draw(rng):
    """One more case of the same uses and ranges (sizes log-uniform, odd ones among them)."""
    use = rng.choice(["lens", "lens", "lens", "batch", "paper", "paper", "synth"])
    precision = rng.choice(["mixed", "fp64"])
    if use == "lens":
        nside = rng.choice([64, 128, 256, 512, 1024, 2048, 4096])
        spin, K = rng.choice([0, 0, 1, 2, 2]), rng.choice([16, 24, 32, 48])
        augmented = spin == 2 and rng.random() < 0.25
        npix = 12 * nside * nside
        most = min(npix, 3e11 / _point_flops(K, spin, augmented) * (1.0 if precision == "mixed" else 0.125))
        count = int(round(10 ** rng.uniform(2.5, math.log10(most))))
        c = _lens("", nside, spin, K, precision, count, augmented=augmented, first=rng.randrange(npix - count + 1),
                  variance=K == 16 and precision == "fp64" and rng.random() < 0.5)
    elif use == "batch":
        c = {"use": "batch", "jobs": rng.randrange(2, 9), "pick": rng.randrange(1 << 20),
             "points": int(round(10 ** rng.uniform(3.0, 4.7)))}
    elif use == "paper":
        nside, y, spin, ss = rng.choice([64, 256, 512, 1024, 2048]), rng.choice([1, 2]), rng.choice([0, 1, 2]), rng.random() < 0.3
        npix = 12 * nside * nside * (4 if ss else 1)
        count = int(round(10 ** rng.uniform(3.0, math.log10(min(npix, 2e7 if y == 1 else 2e6)))))
        c = _paper("", nside, spin, y, precision, count, ss, rng.randrange(npix - count + 1))
    else:
        nside = rng.choice([64, 128, 256, 512])
        c = {"use": "synth", "nside": nside, "lmax": rng.randrange(nside, 2 * nside + 1), "spin": rng.choice([0, 1, 2]),
             "precision": precision}
    c.pop("name", None)
    return c


def _batch_jobs(case):
    """The jobs of a batch: Nside, K and spin as the batched workload draws them, ranges of different lengths."""
    rng = np.random.Generator(np.random.PCG64(case["pick"]))
    jobs = []
    for _ in range(case["jobs"]):
        nside, K, spin = int(rng.choice([256, 512, 1024])), int(rng.choice([16, 24, 32, 48])), int(rng.choice([0, 2]))
        count = max(1, int(case["points"] * rng.uniform(0.25, 1.75)))
        first = int(rng.integers(0, 12 * nside * nside - count + 1))
        jobs.append(_lens("", nside, spin, K, "mixed", count, first=first))
    return jobs


# --------------------------------------------------------------- work per pass
def _point_flops(K, spin, augmented=False):
    """The method's operations per target: assembly of the K x K covariance, its factor, two or three solves."""
    pairs, cm = K * (K - 1) / 2, 4 if spin else 1
    if augmented:
        n = 2 * K
        return 2 * (n ** 3 - n) / 6 + 3 * n * n + pairs * 88 + 6 * n
    return 2 * cm * ((K ** 3 - K) / 6 + 2 * pairs) + pairs * (66 if spin else 16) + 8 * K


def _lens_work(c):
    two = 2 if c["spin"] else 1
    per = 16 + 8 * two + 8 * two + (8 if c["variance"] else 0) + 1  # deflection, source pixel, value, variance, status
    return c["count"] * per, c["count"] * _point_flops(c["K"], c["spin"], c.get("augmented", False))


def work(case):
    use = case["use"]
    if use == "lens":
        b, f = _lens_work(case)
    elif use == "batch":
        parts = [_lens_work(j) for j in _batch_jobs(case)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif use == "paper":
        two, K = 2 if case["spin"] else 1, 9 * 4 ** (case["y"] - 1)
        cm = 4 if case["spin"] else 1
        source = 8 * two * (0.25 if case["supersample"] else 1)
        b = case["count"] * ((0 if case["supersample"] else 16) + source + 8 * two + 8)
        f = case["count"] * (K * (16 + (36 if case["spin"] else 0)) + cm * (2 * K * (K + 1) + 4 * K))
    else:
        n, L = case["nside"], case["lmax"]
        two = 2 if case["spin"] else 1
        b = 16 * two * (L + 1) * (L + 2) / 2 + 8 * two * 12 * n * n
        # per (ring pair, m, l): the recurrence and the sums of both hemispheres
        f = 2 * n * (L + 1) * (L + 2) / 2 * (2 * (3 + 4) if case["spin"] == 0 else 2 * 2 * (3 + 8))
    return {"bytes": float(b), "flops": float(f)}


# --------------------------------------------------- geometry and random fields
def _rings(nside):
    """Per ring 1 .. 4 Nside - 1: z, sin(theta), pixel count, first pixel, azimuth offset (in pixels)."""
    i = torch.arange(1, 4 * nside, dtype=torch.int64, device=DEV)
    m = torch.minimum(i, 4 * nside - i)
    cap, d = m < nside, m.to(F64)
    zc = 1.0 - d * d / (3.0 * nside * nside)
    z = torch.where(cap, torch.where(i < 2 * nside, zc, -zc), (4.0 * nside - 2.0 * i.to(F64)) / (3.0 * nside))
    sc = d * torch.sqrt(6.0 * nside * nside - d * d) / (3.0 * nside * nside)
    e = i.to(F64)
    s = torch.where(cap, sc, torch.sqrt(((2.0 * e - nside) * (7.0 * nside - 2.0 * e)).clamp(min=0)) / (3.0 * nside))
    n = torch.where(cap, 4 * m, torch.full_like(m, 4 * nside))
    first = torch.cumsum(n, 0) - n
    f = torch.where(cap | ((i + nside) % 2 == 0), 0.5, 0.0).to(F64)
    return z, s, n, first, f


def _centres(nside, pix, rings=None):
    """z, sin(theta), cos(phi), sin(phi) of RING pixels."""
    z, s, n, first, f = rings if rings is not None else _rings(nside)
    r = torch.searchsorted(first, pix, right=True) - 1
    phi = ((pix - first[r]).to(F64) + f[r]) * (2.0 * math.pi) / n[r].to(F64)
    return z[r], s[r], torch.cos(phi), torch.sin(phi)


def _cl(lmax, damp, spin):
    """The workloads' spectra: T, 0.05 T for E modes, and l(l+1) C_l^phiphi ~ l^-2 for a deflection field."""
    ell = np.arange(lmax + 1, dtype=np.float64)
    cl = np.zeros(lmax + 1)
    e = ell[2:]
    if spin == 1:
        cl[2:] = e * (e + 1.0) * e ** -4.0
        return cl * (DEFL_RMS ** 2 / np.sum((2.0 * ell + 1.0) / (4.0 * math.pi) * cl))
    cl[2:] = (1e3 if spin == 0 else 50.0) / (e * (e + 1.0)) * np.exp(-((e / damp) ** 2))
    return cl


def _waves(cl, gen):
    """Wave vectors (3, WAVES) with |k| distributed as (2l+1) C_l, phases, and the field's rms."""
    w = (2.0 * np.arange(len(cl)) + 1.0) * cl
    cdf = torch.from_numpy(np.cumsum(w) / np.sum(w))
    ell = torch.searchsorted(cdf, torch.rand(WAVES, generator=gen, dtype=F64)).clamp(max=len(cl) - 1).to(F64)
    u = torch.randn(3, WAVES, generator=gen, dtype=F64)
    u = u / u.norm(dim=0)
    return u.tolist(), ell.tolist(), (2 * math.pi * torch.rand(WAVES, generator=gen, dtype=F64)).tolist(), math.sqrt(np.sum(w) / (4 * math.pi))


def _field(nside, first, count, waves, spin, out=None):
    """The waves' spin-0 field, gradient (spin 1) or traceless second derivative (spin 2) at pixels first .. first + count."""
    u, ell, ph, rms = waves
    out = torch.empty((count,) if spin == 0 else (count, 2), dtype=F64, device=DEV) if out is None else out
    rings = _rings(nside)
    for a in range(0, count, 1 << 24):
        pix = torch.arange(first + a, first + min(a + (1 << 24), count), dtype=torch.int64, device=DEV)
        z, s, c, sn = _centres(nside, pix, rings)
        p = torch.zeros_like(z)
        q = torch.zeros_like(z) if spin else None
        for x, y, w, k, f in zip(*u, ell, ph):
            h = x * c + y * sn
            arg = (h * s + w * z) * k + f
            if spin == 0:
                p += torch.cos(arg)
                continue
            A, B = h * z - w * s, y * c - x * sn  # unit wave vector on e_theta, e_phi
            if spin == 1:
                t = torch.sin(arg)
                p.addcmul_(A, t)
                q.addcmul_(B, t)
            else:
                t = torch.cos(arg)
                p.addcmul_(A * A - B * B, t)
                q.addcmul_(A * B * 2.0, t)
        # mean squares of the factors: cos^2: 1/2; A^2 + B^2: 2/3; (A^2 + B^2)^2: 8/15
        scale = rms / math.sqrt(WAVES * {0: 0.5, 1: 1 / 3, 2: 4 / 15}[spin])
        if spin == 0:
            out[a:a + len(pix)] = p * scale
        else:
            out[a:a + len(pix), 0] = p * scale
            out[a:a + len(pix), 1] = q * scale
    return out


def _gen(seed, k=0):
    return torch.Generator().manual_seed((int(seed) * 1000003 + k) & 0x7FFFFFFFFFFF)


def _inputs(c, seed, k=0):
    """Map and deflections of one lensing job."""
    gen = _gen(seed, k)
    m = _field(c["nside"], 0, 12 * c["nside"] ** 2, _waves(_cl(c["lmax"], c["damp"], c["spin"]), gen), c["spin"])
    if c.get("supersample"):
        return m, None
    return m, _field(c["nside"], c["first"], c["count"], _waves(_cl(c["lmax"], 0.0, 1), gen), 1)


def _alm(lmax, cl, gen):
    a = torch.randn(lmax + 1, lmax + 1, dtype=torch.complex128, generator=gen, device=DEV)
    a *= torch.from_numpy(np.sqrt(cl)).to(DEV)[:, None]
    a = torch.tril(a)
    a[:, 0] = a[:, 0].real * math.sqrt(2.0)
    return a.contiguous()


# -------------------------------------------------------------- prepare and run
def _buffers(c):
    two = (2,) if c["spin"] else ()
    return {"out": torch.empty((c["count"],) + two, dtype=F64, device=DEV),
            "var": torch.empty(c["count"], dtype=F64, device=DEV) if c.get("variance", True) else None,
            "status": torch.empty(c["count"], dtype=torch.uint8, device=DEV)}


def _plan(c):
    return fl.Plan(c["nside"], _cl(c["lmax"], c["damp"], c["spin"]), spin=c["spin"], K=c["K"], precision=c["precision"],
                   flags=fl.FLINTS_SPIN2_AUGMENTED if c["augmented"] else 0)


def prepare(case, seed):
    use = case["use"]
    if use == "lens":
        m, d = _inputs(case, seed)
        return {"use": use, "case": case, "plan": _plan(case), "map": m, "defl": d, **_buffers(case)}
    if use == "batch":
        jobs = []
        for k, c in enumerate(_batch_jobs(case)):
            m, d = _inputs(c, seed, k)
            b = _buffers(c)
            jobs.append((_plan(c), c["first"], c["count"], m, d, b["out"], b["var"], b["status"]))
        return {"use": use, "jobs": jobs, "batch": fl.Batch(len(jobs))}
    if use == "paper":
        m, d = _inputs(case, seed)
        plan = fl.PaperPlan(case["nside"], _cl(case["lmax"], case["damp"], case["spin"]), case["y"], case["precision"],
                            spin=case["spin"])
        return {"use": use, "case": case, "plan": plan, "map": m, "defl": d, **_buffers(case)}
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    cl = _cl(case["lmax"], 0.61 * case["lmax"], case["spin"])
    return {"use": use, "plan": fl.Synth(case["nside"], case["lmax"], case["spin"], case["precision"]),
            "alm": _alm(case["lmax"], cl, gen), "blm": _alm(case["lmax"], 0.1 * cl, gen) if case["spin"] else None,
            "map": torch.empty((12 * case["nside"] ** 2,) + ((2,) if case["spin"] else ()), dtype=F64, device=DEV)}


def run(s):
    if s["use"] == "lens":
        c = s["case"]
        return s["plan"].lens(s["map"], s["defl"], s["out"], s["var"], s["status"], c["first"], c["count"])
    if s["use"] == "batch":
        s["batch"].run(s["jobs"])
        return [j[5:8] for j in s["jobs"]]
    if s["use"] == "paper":
        c = s["case"]
        if c["supersample"]:
            s["plan"].supersample(s["map"], 2 * c["nside"], c["first"], c["count"], s["out"], s["var"], s["status"])
        else:
            s["plan"].lens(s["map"], s["defl"], c["first"], c["count"], s["out"], s["var"], s["status"])
        return s["out"], s["var"], s["status"]
    return s["plan"].run(s["alm"], s["blm"], out=s["map"])


# ------------------------------------------------------------------------ exact
class _Xi:
    """xi (spin 0), xi+ and xi- (spin 1, 2) over xi(0) on t = chord^2 in [0, t_max]: direct sums over l at
    Chebyshev nodes (increments in 1 - cos b, so nothing cancels near b = 0), evaluated by Clenshaw's rule."""

    def __init__(self, cl, spin, t_max):
        nodes = 72
        th = (np.arange(nodes) + 0.5) * math.pi / nodes
        t = np.concatenate([0.5 * t_max * (1.0 + np.cos(th)), [0.0]])
        fp, fm = self._sum(cl, spin, 0.5 * t)
        self.xi0, self.t_max = float(fp[-1]), t_max
        basis = np.cos(np.outer(np.arange(nodes), th)) * (2.0 / nodes)
        basis[0] *= 0.5
        self.plus = (basis @ (fp[:-1] / self.xi0)).tolist()
        self.minus = (basis @ (fm[:-1] / self.xi0)).tolist()

    @staticmethod
    def _sum(cl, spin, u):
        lmax, w = len(cl) - 1, (2.0 * np.arange(len(cl)) + 1.0) / (4.0 * math.pi) * cl
        fp, fm = np.zeros_like(u), np.zeros_like(u)
        s2, x = float(spin * spin), 1.0 - u
        d, inc = (1.0 - 0.5 * u) ** spin, np.zeros_like(u)
        e, em = (0.5 * u) ** spin, np.zeros_like(u)
        for l in range(spin, lmax + 1):
            fp += w[l] * d
            fm += w[l] * e
            if l == 0:
                inc, em, e = -u, e, x
            else:
                den = l * ((l + 1.0) ** 2 - s2)
                a, b, c = (2.0 * l + 1.0) / den, l * (l + 1.0), (l + 1.0) * (l * l - s2) / den
                inc = c * inc - a * b * u * d
                e, em = a * (b * x + s2) * e - c * em, e
            d = d + inc
        return fp, fm

    def __call__(self, t, minus=False):
        c = self.minus if minus else self.plus
        x = t * (2.0 / self.t_max) - 1.0
        b1, b2 = torch.zeros_like(t), torch.zeros_like(t)
        for k in range(len(c) - 1, 0, -1):
            b1, b2 = 2.0 * x * b1 - b2 + c[k], b1
        return x * b1 - b2 + c[0]


def _vec(fr):
    z, s, c, sn = fr
    return torch.stack([s * c, s * sn, z], -1)


def _bases(fr):
    z, s, c, sn = fr
    return torch.stack([z * c, z * sn, -s], -1), torch.stack([-sn, c, torch.zeros_like(c)], -1)


def _angle(d, fr):
    """Projection d.e_theta + i d.e_phi on the local bases."""
    a, b = _bases(fr)
    return torch.complex((d * a).sum(-1), (d * b).sum(-1))


def _targets(nside, first, a, b, defl):
    """Position and frame of targets a .. b of a range, displaced along their deflections."""
    fr = _centres(nside, torch.arange(first + a, first + b, dtype=torch.int64, device=DEV))
    if defl is None:
        return _vec(fr), fr
    d = defl[a:b]
    dl = d.norm(dim=-1, keepdim=True)
    et, ep = _bases(fr)
    n = torch.cos(dl) * _vec(fr) + torch.sinc(dl / math.pi) * (d[:, :1] * et + d[:, 1:] * ep)
    s = torch.hypot(n[:, 0], n[:, 1])
    safe = s.clamp(min=1e-300)
    return n, (n[:, 2], s, torch.where(s > 1e-12, n[:, 0] / safe, 1.0), torch.where(s > 1e-12, n[:, 1] / safe, 0.0))


def _nearest(nside, n, K, rings):
    """The K pixels nearest to each direction: of the rings and azimuths that can hold them, the K smallest chords."""
    z, s, cnt, first, f = rings
    R, W = math.ceil(1.5 * 1.25 * math.sqrt(K / 3.0)) + 2, math.ceil(1.25 * math.sqrt(K / 3.0) / 1.17) + 1
    i0 = torch.searchsorted(-z, -n[:, 2].contiguous())
    r = i0[:, None] + torch.arange(-R, R + 1, device=DEV)
    ok = (r >= 0) & (r < 4 * nside - 1)
    r = r.clamp(0, 4 * nside - 2)
    m = cnt[r]
    phi = torch.atan2(n[:, 1], n[:, 0])[:, None]
    j0 = torch.round(phi * m / (2.0 * math.pi) - f[r]).to(torch.int64)
    o = torch.arange(-W, W + 1, device=DEV)
    j = j0[..., None] + o
    ok = ok[..., None] & (o >= -((m - 1) // 2)[..., None]) & (o <= (m // 2)[..., None])
    pix = (first[r][..., None] + torch.remainder(j, m[..., None])).flatten(1)
    ph = (torch.remainder(j, m[..., None]).to(F64) + f[r][..., None]) * (2.0 * math.pi) / m[..., None].to(F64)
    sr, zr = s[r][..., None], z[r][..., None]
    t = ((sr * torch.cos(ph) - n[:, 0, None, None]) ** 2 + (sr * torch.sin(ph) - n[:, 1, None, None]) ** 2
         + (zr - n[:, 2, None, None]) ** 2)
    t = torch.where(ok, t, torch.full_like(t, 9.0)).flatten(1)
    return torch.gather(pix, 1, torch.topk(t, K, dim=1, largest=False).indices)


def _estimate(nside, n, frn, pix, mp, xi, spin, augmented, rings):
    """Conditional mean and variance from the pixels pix (negative: absent) of each row."""
    absent = pix < 0
    frm = _centres(nside, pix.clamp(min=0), rings)
    X = _vec(frm)
    K = pix.shape[1]
    y = mp[pix.clamp(min=0)]
    d = X[:, None, :, :] - X[:, :, None, :]  # from i (row) to j (column)
    d0 = X - n[:, None, :]
    t, t0 = (d * d).sum(-1), (d0 * d0).sum(-1)
    S, c = xi(t), xi(t0)
    if spin == 0:
        y = y[..., None]
    else:
        fi = tuple(v[:, :, None] for v in frm)
        fj = tuple(v[:, None, :] for v in frm)
        ft = tuple(v[:, None] for v in frn)
        wi, wj, w0, w1 = _angle(d, fi), _angle(d, fj), _angle(d0, ft), _angle(d0, frm)
        unit = lambda q: torch.where(q.abs() > 0, q / q.abs().clamp(min=1e-300), torch.ones_like(q))
        php, ph0 = unit(wi * wj.conj()) ** spin, unit(w0 * w1.conj()) ** spin
        y = torch.complex(y[..., 0], y[..., 1])[..., None]
        if augmented:
            Sm, cm = xi(t, True) * unit(wi * wj) ** 2, xi(t0, True) * unit(w0 * w1) ** 2
            Sm = torch.where(torch.eye(K, dtype=torch.bool, device=DEV), torch.zeros_like(Sm), Sm)
            G, C, g, h = S * php, Sm, c * ph0.conj(), cm
            A = torch.cat([torch.cat([(G + C).real, (C - G).imag], 2), torch.cat([(G + C).imag, (G - C).real], 2)], 1)
            bq, bu = torch.cat([(g + h).real, (g + h).imag], 1), torch.cat([(h - g).imag, (g - h).real], 1)
            x = torch.cat([y.real, y.imag], 1)
            A.diagonal(dim1=1, dim2=2).fill_(1.0 + NUGGET)
            Z = torch.linalg.solve_triangular(torch.linalg.cholesky(A), torch.cat([bq[..., None], bu[..., None], x], 2), upper=False)
            q, u, zx = Z.unbind(2)
            v = torch.stack([(q * zx).sum(1), (u * zx).sum(1)], 1)
            return v, xi.xi0 * (1.0 - 0.5 * ((q * q).sum(1) + (u * u).sum(1)))
        S, c = S * php, (c * ph0).conj()
    if bool(absent.any()):
        S = S.masked_fill(absent[:, :, None] | absent[:, None, :], 0.0)
        c, y = c.masked_fill(absent, 0.0), y.masked_fill(absent[..., None], 0.0)
    S.diagonal(dim1=1, dim2=2).fill_(1.0 + NUGGET)
    Z = torch.linalg.solve_triangular(torch.linalg.cholesky(S), torch.cat([c[..., None], y], 2), upper=False)
    zc, zy = Z[..., 0], Z[..., 1]
    v, q = (zc.conj() * zy).sum(1), (zc.abs() ** 2).sum(1)
    return (torch.stack([v.real, v.imag], 1) if spin else v), xi.xi0 * (1.0 - q)


def _exact_lens(c, mp, defl):
    nside, spin, K = c["nside"], c["spin"], c["K"]
    rings = _rings(nside)
    xi = _Xi(_cl(c["lmax"], c["damp"], spin), spin, 4.0 * (1.25 ** 2) * (K / 3.0) / nside ** 2)
    b = _buffers(c)
    step = max(1, (1 << 25) // (K * K * (4 if c["augmented"] else 1)))
    for a in range(0, c["count"], step):
        e = min(a + step, c["count"])
        n, fr = _targets(nside, c["first"], a, e, defl)
        pix = _nearest(nside, n, K, rings)
        b["out"][a:e], v = _estimate(nside, n, fr, pix, mp, xi, spin, c["augmented"], rings)
        if c["variance"]:
            b["var"][a:e] = v
    return b["out"], b["var"], torch.zeros_like(b["status"])


# The paper's stencil: the pixel that holds the target on the grid Nside / 2^(y-1), the pixels that share a vertex
# with it, and their children.  Pixels are cells (a, b) .. (a + 1, b + 1) of a quadrant's cap coordinates or diamonds
# of the belt; a cell's corners are compared as points on the sphere.
def _corners(nside, pix, rings):
    z, s, n, first, f = rings
    N = float(nside)
    r = torch.searchsorted(first, pix, right=True) - 1
    i = r + 1
    m = torch.minimum(i, 4 * nside - i)
    south = i > 2 * nside
    j = pix - first[r]
    phi = (j.to(F64) + f[r]) * (2.0 * math.pi) / n[r].to(F64)

    def cap(a, b, q):  # point of quadrant q's cap coordinates
        h = a + b
        az = (q + a / h.clamp(min=1e-9)) * (0.5 * math.pi)
        zz = 1.0 - (h / N) ** 2 / 3.0
        ss = (h / N) * torch.sqrt((2.0 - (h / N) ** 2 / 3.0) / 3.0)
        return torch.stack([ss * torch.cos(az), ss * torch.sin(az), torch.where(south, -zz, zz)], -1)

    def belt(zz, az):
        ss = torch.sqrt((1.0 - zz * zz).clamp(min=0))
        return torch.stack([ss * torch.cos(az), ss * torch.sin(az), zz], -1)

    polar = (m <= nside)[..., None]
    mm = torch.minimum(m, torch.full_like(m, nside))
    q = torch.div(j, mm, rounding_mode="floor").to(F64)
    # ring m of the cap, its k-th cell: a = k, b = m - 1 - k (ring Nside is shifted like the cap's: offset 1/2)
    k = (j - torch.div(j, mm, rounding_mode="floor") * mm).to(F64)
    a, b = k, (mm - 1).to(F64) - k
    dz, dp = 2.0 / (3.0 * N), 0.25 * math.pi / N
    zr = z[r]
    inner_cap, inner_belt = cap(a, b, q), belt(torch.where(south, zr - dz, zr + dz), phi)
    east = torch.where(polar, cap(a + 1, b, q), belt(zr, phi + dp))
    west = torch.where(polar, cap(a, b + 1, q), belt(zr, phi - dp))
    outer_cap, outer_belt = cap(a + 1, b + 1, q), belt(torch.where(south, zr + dz, zr - dz), phi)
    outer = torch.where((m < nside)[..., None], outer_cap, outer_belt)
    return torch.stack([torch.where(polar, inner_cap, inner_belt), east, west, outer], -2)


def _locate(nside, n, rings):
    """RING pixel that holds each direction."""
    z, s, cnt, first, f = rings
    N = float(nside)
    x, za = n[:, 2], n[:, 2].abs()
    tt = torch.remainder(torch.atan2(n[:, 1], n[:, 0]) * (2.0 / math.pi), 4.0)
    jp = torch.floor(N * (0.5 + tt) - 0.75 * N * x)
    jm = torch.floor(N * (0.5 + tt) + 0.75 * N * x)
    ring = nside + 1 + (jp - jm).to(torch.int64)  # 1 .. 2 Nside + 1 from z = 2/3
    shift = 1 - (ring & 1)
    ip = torch.remainder(torch.div(((jp + jm).to(torch.int64) - nside + shift + 1), 2, rounding_mode="floor"), 4 * nside)
    belt = 2 * nside * (nside - 1) + (ring - 1) * 4 * nside + ip
    tp = tt - torch.floor(tt)
    h = N * torch.hypot(n[:, 0], n[:, 1]) * torch.sqrt(3.0 / (1.0 + za))
    ir = (torch.floor(tp * h) + torch.floor((1.0 - tp) * h)).to(torch.int64) + 1
    ip = torch.remainder(torch.floor(tt * ir).to(torch.int64), 4 * ir)
    polar = torch.where(x > 0, 2 * ir * (ir - 1) + ip, 12 * nside * nside - 2 * ir * (ir + 1) + ip)
    return torch.where(za <= 2.0 / 3.0, belt, polar)


def _vertex_stencil(nside, pix, rings):
    """The pixels that share a vertex with pix, itself among them: (B, 9), -1 where there are fewer."""
    z, s, cnt, first, f = rings
    r0 = torch.searchsorted(first, pix, right=True) - 1
    phi = ((pix - first[r0]).to(F64) + f[r0]) / cnt[r0].to(F64)
    r = r0[:, None] + torch.arange(-2, 3, device=DEV)
    ok = (r >= 0) & (r < 4 * nside - 1)
    r = r.clamp(0, 4 * nside - 2)
    m = cnt[r]
    o = torch.arange(-3, 4, device=DEV)
    j = torch.round(phi[:, None] * m - f[r]).to(torch.int64)[..., None] + o
    ok = ok[..., None] & (o >= -((m - 1) // 2)[..., None]) & (o <= (m // 2)[..., None])
    cand = torch.where(ok, first[r][..., None] + torch.remainder(j, m[..., None]), 0).flatten(1)
    ok = ok.flatten(1)
    own, other = _corners(nside, pix, rings), _corners(nside, cand, rings)
    near = torch.zeros_like(ok)
    for k in range(4):
        near |= ((other - own[:, None, None, k, :]).abs().amax(-1) < 0.01 / nside).any(-1)
    near &= ok
    pos = torch.cumsum(near, 1) - 1
    out = torch.full((len(pix), 10), -1, dtype=torch.int64, device=DEV)
    out.scatter_(1, torch.where(near, pos, 9), torch.where(near, cand, -1))
    return out[:, :9]


def _children(nside, pix, rings, fine_rings):
    """The four pixels of the grid 2 Nside inside each pixel: those that hold points a third of the way to its corners."""
    safe = pix.clamp(min=0)
    c = _corners(nside, safe, rings)
    mid = _vec(_centres(nside, safe, rings))
    p = mid[..., None, :] + 0.3 * (c - mid[..., None, :])
    p = p / p.norm(dim=-1, keepdim=True)
    ch = _locate(2 * nside, p.reshape(-1, 3), fine_rings).reshape(pix.shape + (4,))
    return torch.where((pix < 0)[..., None], -1, ch).flatten(1)


def _exact_paper(c, mp, defl):
    nside, spin, y = c["nside"], c["spin"], c["y"]
    coarse = nside >> (y - 1)
    rings, crings = _rings(nside), _rings(coarse)
    xi = _Xi(_cl(c["lmax"], c["damp"], spin), spin, min((7.0 / coarse) ** 2, 4.0))
    b = _buffers(c)
    step = 1 << (20 if y == 1 else 15)
    for a in range(0, c["count"], step):
        e = min(a + step, c["count"])
        n, fr = _targets(2 * nside if defl is None else nside, c["first"], a, e, defl)
        pix = _vertex_stencil(coarse, _locate(coarse, n, crings), crings)
        if y == 2:
            pix = _children(coarse, pix, crings, rings)
        b["out"][a:e], b["var"][a:e] = _estimate(nside, n, fr, pix, mp, xi, spin, False, rings)
    return b["out"], b["var"], torch.zeros_like(b["status"])


def _exact_synth(case, alm, blm):
    """P = -sum (E + iB) sY_lm (spin 0: sum a Y), F_m per ring by the Wigner-d recurrence in l, then a DFT per ring."""
    N, L, s = case["nside"], case["lmax"], case["spin"]
    z = _rings(N)[0][:2 * N]
    lc, ls = 0.5 * torch.log2((1.0 + z) / 2.0), 0.5 * torch.log2((1.0 - z) / 2.0)
    m = torch.arange(L + 1, device=DEV, dtype=F64)
    lg = lambda v: torch.lgamma(v + 1.0)
    cols = []
    for sg in ((0,) if s == 0 else (-s, s)):  # d_{m, sg}
        hi = m.clamp(min=s)
        # m >= s: d^m_{m,sg}: (-1)^(m-sg) c^(m+sg) s^(m-sg);  m < s: d_{m,-s} = d_{s,-m}: (-1)^(s+m) c^(s-m) s^(s+m),
        # d_{m,s} = d_{-s,-m}: c^(s+m) s^(s-m)
        pc = torch.where(m >= s, m + sg, s - m if sg < 0 else s + m)
        ps = torch.where(m >= s, m - sg, s + m if sg < 0 else s - m)
        neg = torch.where(m >= s, torch.remainder(m - sg, 2.0), torch.remainder(s + m, 2.0) if sg < 0 else torch.zeros_like(m))
        amp = 0.5 * (lg(2.0 * hi) - lg(pc) - lg(ps)) / math.log(2.0)
        e = amp + pc * lc[:, None] + ps * ls[:, None]
        E = torch.floor(e)
        cols.append([torch.exp2(e - E) * (1.0 - 2.0 * neg), torch.zeros_like(e), E, sg])
    shape = (2 * N, L + 1)
    acc = {(k, w, p): torch.zeros(shape, dtype=torch.complex128, device=DEV)
           for k in range(len(cols)) for w in range(1 if s == 0 else 2) for p in (0, 1)}
    for l in range(s, L + 1):
        M = l + 1  # columns with l0 <= l
        nl = math.sqrt((2.0 * l + 1.0) / (4.0 * math.pi))
        if s == 0:
            ws = [alm[l, :M] * nl]
        else:
            ws = [(alm[l, :M] + 1j * blm[l, :M]) * nl, (alm[l, :M].conj() + 1j * blm[l, :M].conj()) * nl]
        par = torch.remainder(l + m[:M], 2.0)
        mm = m[:M]
        for k, col in enumerate(cols):
            v, p, E = col[0][:, :M], col[1][:, :M], col[2][:, :M]
            d = torch.ldexp(v, E.clamp(min=-1000))
            for w, wt in enumerate(ws):
                acc[k, w, 0][:, :M] += d * (wt * (1.0 - par))
                acc[k, w, 1][:, :M] += d * (wt * par)
            if l == L:
                continue
            if l == 0:
                A, B, C = torch.ones_like(mm), torch.zeros_like(mm), torch.zeros_like(mm)
            else:
                den = l * torch.sqrt(((l + 1.0) ** 2 - mm * mm) * ((l + 1.0) ** 2 - s * s))
                A = (2.0 * l + 1.0) * l * (l + 1.0) / den
                B = (2.0 * l + 1.0) * mm * col[3] / den
                C = (l + 1.0) * torch.sqrt((l * l - mm * mm).clamp(min=0) * (l * l - s * s)) / den
            nv = (A * z[:, None] - B) * v - C * p
            col[1][:, :M] = v
            col[0][:, :M] = nv
            if l % 8 == 0:
                big = nv.abs() > 2.0 ** 200
                col[0][:, :M] = torch.where(big, nv * 2.0 ** -200, nv)
                col[1][:, :M] = torch.where(big, col[1][:, :M] * 2.0 ** -200, col[1][:, :M])
                col[2][:, :M] = torch.where(big, E + 200.0, E)
    tot = lambda k, w, sg: acc[k, w, 0] + sg * acc[k, w, 1]
    if s == 0:
        north, south = [tot(0, 0, 1), None], [tot(0, 0, -1), None]
    else:
        sg = 1.0 if s % 2 else -1.0
        north = [sg * tot(0, 0, 1), -tot(1, 1, 1)]
        south = [sg * tot(1, 0, -1), -tot(0, 1, -1)]
    out = torch.empty((12 * N * N, 2) if s else 12 * N * N, dtype=F64, device=DEV)
    mi = torch.arange(L + 1, device=DEV)
    for i in range(1, 4 * N):
        mirror = min(i, 4 * N - i)
        n = 4 * min(mirror, N)
        src, row = (north, i - 1) if i <= 2 * N else (south, mirror - 1)
        half = 0.5 if mirror < N or (i + N) % 2 == 0 else 0.0
        ph = torch.exp(1j * (2.0 * math.pi * half / n) * m)
        H = torch.zeros(n, dtype=torch.complex128, device=DEV)
        a = src[0][row] * ph
        H.index_add_(0, mi % n, a)
        nega = (a.conj() if s == 0 else src[1][row] * ph.conj())[1:]
        H.index_add_(0, (-mi[1:]) % n, nega)
        x = torch.fft.ifft(H, norm="forward")
        st = 2 * i * (i - 1) if i < N else (2 * N * (N - 1) + 4 * N * (i - N) if i <= 3 * N else 12 * N * N - 2 * mirror * (mirror + 1))
        if s == 0:
            out[st:st + n] = x.real
        else:
            out[st:st + n, 0], out[st:st + n, 1] = x.real, x.imag
    return out


def exact(case, seed):
    use = case["use"]
    if use == "lens":
        return _exact_lens(case, *_inputs(case, seed))
    if use == "batch":
        return [_exact_lens(c, *_inputs(c, seed, k)) for k, c in enumerate(_batch_jobs(case))]
    if use == "paper":
        return _exact_paper(case, *_inputs(case, seed))
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    cl = _cl(case["lmax"], 0.61 * case["lmax"], case["spin"])
    alm = _alm(case["lmax"], cl, gen)
    return _exact_synth(case, alm, _alm(case["lmax"], 0.1 * cl, gen) if case["spin"] else None)
