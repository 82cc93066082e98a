"""Timed cases of the spherical harmonic transforms, through the package's public entry points.

``listed()`` gives the fixed cases, ``draw(rng)`` more of the same ranges.  A case names a path
("what"), a grid, the band limits and the number of maps; ``prepare`` makes the plan a program keeps
and inputs drawn on the GPU from the seed, ``run`` makes one call (or the two of a round trip),
``work`` states what one pass cannot do without and ``exact`` evaluates the same sums with plain
torch in 64 bits, on a geometry that is computed here.

Paths: "synth" / "anal" (alm2map / map2alm), "round" (alm2map, then map2alm of its maps), "spin_synth" /
"spin_anal" (E, B <-> Q, U) and "batch" (many FP64 transforms of uneven band limits and both
directions as one PersistentBatch).  mode "fp64" is the default arithmetic of a plan, "split" the
precision form.  HEALPix cases have mmax = lmax.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1106_0159_gb300 import batch, sht

MODES = {"fp64": sht.MODE_FP64, "split": sht.MODE_SPLIT_BF16}


def _hp(what, nside, lmax, maps, mode="fp64"):
    return {"what": what, "grid": "healpix", "nside": nside, "lmax": lmax, "mmax": lmax, "maps": maps, "mode": mode}


def _gl(what, rings, nphi, lmax, mmax, maps, mode="fp64"):
    return {"what": what, "grid": "gl", "rings": rings, "nphi": nphi, "lmax": lmax, "mmax": mmax, "maps": maps,
            "mode": mode}


def listed():
    named = {
        # the smallest benchmark configuration, one map at a time: launches and latency count
        "synth_small": _hp("synth", 32, 64, 1),
        "anal_small": _hp("anal", 32, 64, 1),
        # one large map in the default arithmetic: interactive use
        "synth_one_map": _hp("synth", 1024, 2048, 1),
        "anal_one_map": _hp("anal", 1024, 2048, 1),
        # a Gauss-Legendre grid with odd sizes, mmax below lmax and a few maps
        "synth_gl_odd": _gl("synth", 751, 1501, 750, 500, 5),
        # several full-size maps in the default arithmetic: spectra of a small ensemble
        "anal_ensemble": _hp("anal", 2048, 4096, 4),
        # the headline workload in the precision form: Monte Carlo batches of 16 full-size maps
        "synth_mc_split": _hp("synth", 2048, 4096, 16, "split"),
        "anal_mc_split": _hp("anal", 2048, 4096, 16, "split"),
        # one request of a transform service: a round trip at an uneven band limit and map count
        "round_served_split": _hp("round", 338, 676, 5, "split"),
        # polarisation maps, each direction
        "spin_synth": _hp("spin_synth", 512, 1024, 1),
        "spin_anal": _hp("spin_anal", 512, 1024, 2),
        # many requests of uneven band limits, both directions, as one persistent batch
        "batch_mixed": {"what": "batch", "lmax": 620, "jobs": 8, "most": 4},
    }
    return [dict(c, name=n) for n, c in named.items()]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    what = rng.choice(["synth", "anal", "synth", "anal", "round", "spin_synth", "spin_anal", "batch"])
    if what == "batch":
        return {"what": what, "lmax": _log(rng, 150, 800), "jobs": rng.randint(3, 9), "most": rng.randint(1, 5)}
    maps = rng.choice([1, 1, 2, 3, 5, 8, 11, 16])
    if what.startswith("spin"):
        mode, maps, top = "fp64", min(maps, 3), 1100
    else:
        mode = rng.choice(["fp64", "split"])
        top = 2048 if mode == "fp64" else 3000
        if what == "round" or maps > 4:
            top = 3 * top // 5
    lmax = _log(rng, 60, top)
    if rng.random() < 0.65:
        return _hp(what, (lmax + 1) // 2, lmax, maps, mode)
    mmax = lmax if rng.random() < 0.6 else rng.randint(lmax // 2, lmax)
    return _gl(what, lmax + rng.randint(1, 4), 2 * mmax + rng.randint(1, 9), lmax, mmax, maps, mode)


# ---------------------------------------------------------------- geometry and inputs

def _healpix(nside):
    i = np.arange(1, 4 * nside)
    north = np.where(i <= 2 * nside, i, 4 * nside - i).astype(np.float64)
    cap = north < nside
    nphi = np.where(cap, 4 * north, 4 * nside).astype(np.int64)
    belt = np.clip(4.0 / 3.0 - 2.0 * north / (3.0 * nside), -1.0, 1.0)
    theta = np.where(cap, 2.0 * np.arcsin(np.minimum(north / (math.sqrt(6.0) * nside), 1.0)), np.arccos(belt))
    theta = np.where(i > 2 * nside, math.pi - theta, theta)
    shift = np.where((i - nside) % 2 == 0, math.pi / (4.0 * nside), 0.0)
    phi0 = np.where(cap, math.pi / (4.0 * north), shift)
    return nphi, theta, phi0, np.full(len(i), 4.0 * math.pi / (12.0 * nside * nside))


def _gauss_legendre(n, nphi):
    th = math.pi * (np.arange((n + 1) // 2) + 0.75) / (n + 0.5)
    for _ in range(8):  # Newton on P_n(cos theta) in theta, by Reinsch's difference form near the pole
        u, s = 2.0 * np.sin(0.5 * th) ** 2, np.sin(th)
        p, q, d = 1.0 - u, np.ones_like(u), -u
        for l in range(1, n):
            d = (l * d - (2.0 * l + 1.0) * u * p) / (l + 1.0)
            q, p = p, p + d
        th = th + p * s / (n * (q - (1.0 - u) * p))
    if n % 2:
        th[-1] = 0.5 * math.pi
    w = 2.0 * math.pi / nphi * 2.0 * s ** 2 / (n * q) ** 2
    south = slice(None, None, -1) if n % 2 == 0 else slice(-2, None, -1)
    return (np.full(n, nphi, np.int64), np.concatenate([th, math.pi - th[south]]), np.zeros(n),
            np.concatenate([w, w[south]]))


def _geometry(case):
    return _healpix(case["nside"]) if case["grid"] == "healpix" else _gauss_legendre(case["rings"], case["nphi"])


def _nalm(lmax, mmax):
    return (mmax + 1) * (lmax + 1) - mmax * (mmax + 1) // 2


def _red_alm(shape, lmax, mmax, gen):
    """CMB-like coefficients: variance 1 / (l (l + 1) + 1), a_l0 real."""
    m = torch.repeat_interleave(torch.arange(mmax + 1, device="cuda"),
                                torch.arange(lmax + 1, lmax - mmax, -1, device="cuda"))
    l = torch.arange(len(m), device="cuda") - m * (2 * lmax + 3 - m) // 2 + m
    sd = torch.rsqrt((l * (l + 1) + 1).double() * torch.where(m == 0, 1.0, 2.0))
    a = torch.randn(shape + (len(m), 2), dtype=torch.float64, device="cuda", generator=gen) * sd[:, None]
    a[..., :lmax + 1, 1] = 0.0
    a = torch.view_as_complex(a)
    return a, l


def _inputs(case, seed):
    gen = torch.Generator("cuda").manual_seed(int(seed))
    n, L, M, what = case["maps"], case["lmax"], case["mmax"], case["what"]
    if what in ("synth", "round"):
        return _red_alm((n,), L, M, gen)[0]
    if what == "spin_synth":
        a, l = _red_alm((n, 2), L, M, gen)
        return a * (l >= 2)
    npix = int(_geometry(case)[0].sum())
    shape = (n, npix) if what == "anal" else (n, 2, npix)
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)


def _batch_jobs(case):
    """The transforms of a batch case, each a case of its own: band limits from lmax / 3 up, both directions."""
    k = case["jobs"]
    out = []
    for j in range(k):
        lmax = round(case["lmax"] * (1 + 2 * j / (k - 1)) / 3)
        out.append(_hp("synth" if j % 2 else "anal", (lmax + 1) // 2, lmax, 1 + 7 * j % case["most"]))
    return out


def _plan(case):
    grid = sht.GRID_HEALPIX if case["grid"] == "healpix" else sht.GRID_GAUSS_LEGENDRE
    plan = sht.Plan(_geometry(case), case["lmax"], case["mmax"], grid=grid)
    if case["mode"] != "fp64":
        plan.set_mode(MODES[case["mode"]])
    return plan


def prepare(case, seed):
    if case["what"] != "batch":
        return {"case": case, "plan": _plan(case), "x": _inputs(case, seed)}
    jobs = []
    for j, c in enumerate(_batch_jobs(case)):
        plan, x = _plan(c), _inputs(c, seed + j)
        if c["what"] == "synth":
            out = torch.empty((c["maps"], plan.npix), dtype=torch.float64, device="cuda")
            jobs.append(batch.Job(plan, batch.ALM2MAP, x, out))
        else:
            out = torch.empty((c["maps"], plan.nalm), dtype=torch.complex128, device="cuda")
            jobs.append(batch.Job(plan, batch.MAP2ALM, x, out))
    return {"case": case, "jobs": jobs, "batch": batch.PersistentBatch(jobs).capture()}


def run(state):
    what = state["case"]["what"]
    if what == "batch":
        state["batch"].replay()
        return [j.dst for j in state["jobs"]]
    plan, x = state["plan"], state["x"]
    if what == "synth":
        return plan.alm2map(x)
    if what == "anal":
        return plan.map2alm(x)
    if what == "round":
        maps = plan.alm2map(x)
        return [maps, plan.map2alm(maps)]
    return plan.alm2map_spin(x) if what == "spin_synth" else plan.map2alm_spin(x)


# ---------------------------------------------------------------- work

def work(case):
    """Coefficients and maps once each; 3 operations of the recurrence per (l, m, ring pair), 4 of the
    sum over l (or over rings) per map, 2.5 n log2 n per ring of n pixels."""
    if case["what"] == "batch":
        each = [work(c) for c in _batch_jobs(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    nphi = _geometry(case)[0]
    n, nalm, npix = case["maps"], _nalm(case["lmax"], case["mmax"]), int(nphi.sum())
    steps = nalm * ((len(nphi) + 1) // 2)
    fft = float(np.sum(2.5 * nphi * np.log2(np.maximum(nphi, 2))))
    passes = 2 if case["what"] == "round" else 1
    if case["what"].startswith("spin"):
        return {"bytes": 2 * n * (16 * nalm + 8 * npix), "flops": steps * (8 + 16 * n) + 2 * n * fft}
    return {"bytes": passes * n * (16 * nalm + 8 * npix), "flops": passes * (steps * (3 + 4 * n) + n * fft)}


# ---------------------------------------------------------------- the same sums in plain torch

BIG = 512   # lambda is kept as value * 2^(BIG k), k <= 0; terms with k < 0 are below 2^-200 and left out
PAD = 16    # steps between two tests of the scale


def _start(m, s, half_s, half_c):
    """(value, exponent) factors that take the start value of m - 1 to that of m (None: from scratch)."""
    if s == 0:
        if m == 0:
            return None, torch.full_like(half_s, math.sqrt(0.25 / math.pi))
        return math.sqrt((2 * m + 1) / (2 * m)), 2.0 * half_s * half_c
    up, dn = (half_s, half_c) if s > 0 else (half_c, half_s)
    if m == 0:
        return None, math.sqrt(7.5 / math.pi) * (half_s * half_c) ** 2
    if m == 1:
        sign = 1.0 if s > 0 else -1.0
        return None, sign * math.sqrt(5.0 / math.pi) * up ** 3 * dn
    if m == 2:
        return None, math.sqrt(1.25 / math.pi) * up ** 4
    return math.sqrt(2 * m * (2 * m + 1) / ((m + 2) * (m - 2))), half_s * half_c


def _columns(lmax, mmax, theta, s):
    """For l = |s| .. lmax: (l, slambda_lm(theta)) for m = 0 .. min(l, mmax), [m, theta]."""
    half_s, half_c = torch.sin(0.5 * theta), torch.cos(0.5 * theta)
    u = 2.0 * half_s ** 2
    P, dev = len(theta), theta.device
    a, b = (torch.zeros((mmax + 1, P), dtype=torch.float64, device=dev) for _ in range(2))
    k = torch.zeros((mmax + 1, P), dtype=torch.int32, device=dev)
    live = torch.ones((mmax + 1, P), dtype=torch.float64, device=dev)
    ms = torch.arange(mmax + 1, dtype=torch.float64, device=dev)
    val, ex = torch.ones_like(theta), torch.zeros_like(theta)
    for l in range(abs(s), lmax + 1):
        rows = min(l, mmax) + 1
        old = min(l - 1, mmax) + 1 if l > abs(s) else 0
        if old:
            m, q = ms[:old, None], float(l - 1)
            A = l * math.sqrt((2 * q + 1) * (2 * q + 3)) / torch.sqrt((l * l - m * m) * (l * l - s * s))
            a1 = a[:old]
            t = a1 - u * a1
            if s and q:
                t.addcmul_(a1, m * (s / (q * l)))
            t *= A
            if q:
                B = torch.sqrt(((q * q - m * m) * (q * q - s * s)).clamp_(min=0.0)) / (q * math.sqrt(4 * q * q - 1))
                t.addcmul_(b[:old], A * B, value=-1.0)
            b[:old], a[:old] = a1, t
        for m in range(old, rows):  # the columns that start at this l
            ratio, f = _start(m, s, half_s, half_c)
            val, ex = (f, torch.zeros_like(ex)) if ratio is None else (val * (ratio * f), ex)
            mant, e = torch.frexp(val)
            val, ex = mant, ex + e
            k[m] = -((-ex).clamp(min=0) // BIG).int()
            a[m] = torch.ldexp(val, ex - BIG * k[m])
            live[m] = (k[m] == 0).double()
        if l % PAD == 0:
            up = (k[:rows] < 0) & (torch.maximum(a[:rows].abs(), b[:rows].abs()) > 2.0 ** (BIG // 2))
            scale = torch.ones_like(a[:rows]).masked_fill_(up, 2.0 ** -BIG)
            a[:rows] *= scale
            b[:rows] *= scale
            k[:rows] += up
            live[:rows] = (k[:rows] == 0).double()
        yield l, a[:rows] * live[:rows]


def _index(l, rows, lmax):
    m = torch.arange(rows, device="cuda")
    return m * (2 * lmax + 3 - m) // 2 + l - m


def _reals(z):
    """[c, m] complex -> [m, 2 c] float: re and im of every channel."""
    return torch.view_as_real(z.t().contiguous()).flatten(1)


def _phase(phi0, mmax):
    """exp(i m phi0), [ring, m], with m phi0 reduced modulo 2 pi in parts."""
    m = torch.arange(mmax + 1, dtype=torch.float64, device="cuda")
    p = torch.from_numpy(phi0).cuda()[:, None]
    p1 = p.float().double()
    p1 = (p1 * 2.0 ** 24).round() / 2.0 ** 24
    c1, c2 = 6.28318500518798828125, 3.019915981956752868e-7  # 2 pi = c1 + c2 to 1e-22; q c1 is exact
    q = torch.round(m * p / (2.0 * math.pi))
    r = ((m * p1 - q * c1) - q * c2) + m * (p - p1)
    return torch.polar(torch.ones_like(r), r)


def _ring_groups(nphi):
    for n in np.unique(nphi):
        yield int(n), torch.from_numpy(np.nonzero(nphi == n)[0]).cuda()


def _to_maps(delta, geom):
    """Ring synthesis of delta [c, ring, m] into maps [c, pixel]."""
    nphi, _, phi0, _ = geom
    ofs = torch.from_numpy(np.concatenate([[0], np.cumsum(nphi)])).cuda()
    C, _, M1 = delta.shape
    out = torch.empty((C, int(nphi.sum())), dtype=torch.float64, device="cuda")
    two = torch.full((M1,), 2.0, dtype=torch.float64, device="cuda")
    two[0] = 1.0
    for n, rings in _ring_groups(nphi):
        v = delta[:, rings] * (_phase(phi0[rings.cpu().numpy()], M1 - 1) * two)
        fold = torch.zeros((C, len(rings), n), dtype=torch.complex128, device="cuda")
        for m0 in range(0, M1, n):
            part = v[..., m0:m0 + n]
            fold[..., :part.shape[-1]] += part
        s = torch.fft.ifft(fold, norm="forward").real
        out[:, (ofs[rings][:, None] + torch.arange(n, device="cuda")).flatten()] = s.flatten(1)
    return out


def _to_delta(maps, geom, mmax):
    """Weighted ring analysis of maps [c, pixel] into [c, ring, m]."""
    nphi, _, phi0, w = geom
    ofs = torch.from_numpy(np.concatenate([[0], np.cumsum(nphi)])).cuda()
    delta = torch.empty((maps.shape[0], len(nphi), mmax + 1), dtype=torch.complex128, device="cuda")
    m = torch.arange(mmax + 1, device="cuda")
    for n, rings in _ring_groups(nphi):
        h = rings.cpu().numpy()
        s = maps[:, ofs[rings][:, None] + torch.arange(n, device="cuda")]
        f = torch.fft.fft(s)[..., m % n]
        delta[:, rings] = f * (_phase(phi0[h], mmax).conj() * torch.from_numpy(w[h]).cuda()[:, None])
    return delta


def _exact_synth(alm, geom, lmax, mmax, spin):
    nr, P = len(geom[1]), (len(geom[1]) + 1) // 2
    theta = torch.from_numpy(geom[1][:P]).cuda()
    C = alm.shape[0]

    def sums():  # [parity of l - m][m, 2 C, slot]
        return torch.zeros((2, mmax + 1, 2 * C, P), dtype=torch.float64, device="cuda")

    def add(acc, l, rows, z, lam):
        c = _reals(z)
        c[0, 1::2] = 0.0  # Im a_l0 is ignored
        for p in (0, 1):
            r = slice((l + p) % 2, rows, 2)
            acc[p, r].addcmul_(c[r, :, None], lam[r, None, :])

    def rings(acc, odd):  # north and south rings from the parity sums
        north, south = acc[0] + acc[1], odd * (acc[0] - acc[1])
        both = torch.cat([north, south.flip(2)[..., (2 * P - nr):]], dim=2)  # an equator ring counts once
        return torch.view_as_complex(both.view(mmax + 1, C, 2, nr).permute(1, 3, 0, 2).contiguous())

    if not spin:
        acc = sums()
        for l, lam in _columns(lmax, mmax, theta, 0):
            add(acc, l, len(lam), alm[:, _index(l, len(lam), lmax)], lam)
        return _to_maps(rings(acc, 1.0), geom)
    swap = alm.view(-1, 2, alm.shape[1]).flip(1).reshape(alm.shape)
    aw, ax = sums(), sums()
    for (l, lp), (_, lm) in zip(_columns(lmax, mmax, theta, 2), _columns(lmax, mmax, theta, -2)):
        ix = _index(l, len(lp), lmax)
        add(aw, l, len(lp), alm[:, ix], 0.5 * (lp + lm))
        add(ax, l, len(lp), swap[:, ix], 0.5 * (lp - lm))
    w, x = rings(aw, 1.0), rings(ax, -1.0)
    delta = torch.empty_like(w)
    delta[0::2] = -(w[0::2] + 1j * x[0::2])   # Delta^Q = -sum (E W + i B X)
    delta[1::2] = -(w[1::2] - 1j * x[1::2])   # Delta^U = -sum (B W - i E X)
    return _to_maps(delta, geom)


def _exact_anal(maps, geom, lmax, mmax, spin):
    nr, P = len(geom[1]), (len(geom[1]) + 1) // 2
    theta = torch.from_numpy(geom[1][:P]).cuda()
    C = maps.shape[0]
    d = _to_delta(maps, geom, mmax)
    north, south = d[:, :P], torch.zeros_like(d[:, :P])
    south[:, :nr - P] = d[:, P:].flip(1)

    def rows_of(z):  # [m, 2 C, slot]
        return torch.view_as_real(z.permute(2, 0, 1)).permute(0, 1, 3, 2).reshape(mmax + 1, 2 * C, P)

    plus, minus = rows_of(north + south), rows_of(north - south)
    out = torch.zeros((C, _nalm(lmax, mmax)), dtype=torch.complex128, device="cuda")

    def dot(l, lam, even, odd):
        rows = len(lam)
        got = torch.empty((rows, 2 * C), dtype=torch.float64, device="cuda")
        for p, x in ((0, even), (1, odd)):
            r = slice((l + p) % 2, rows, 2)
            got[r] = torch.bmm(x[r], lam[r, :, None])[..., 0]
        return torch.view_as_complex(got.view(rows, C, 2)).t()

    if not spin:
        for l, lam in _columns(lmax, mmax, theta, 0):
            out[:, _index(l, len(lam), lmax)] = dot(l, lam, plus, minus)
    else:
        for (l, lp), (_, lm) in zip(_columns(lmax, mmax, theta, 2), _columns(lmax, mmax, theta, -2)):
            w = dot(l, 0.5 * (lp + lm), plus, minus)
            x = dot(l, 0.5 * (lp - lm), minus, plus)
            e = torch.empty_like(w)
            e[0::2] = -(w[0::2] + 1j * x[1::2])
            e[1::2] = 1j * x[0::2] - w[1::2]
            out[:, _index(l, len(lp), lmax)] = e
    out[:, :lmax + 1] = out[:, :lmax + 1].real.to(torch.complex128)
    return out


def exact(case, seed):
    if case["what"] == "batch":
        return [exact(c, seed + j) for j, c in enumerate(_batch_jobs(case))]
    geom, x, what = _geometry(case), _inputs(case, seed), case["what"]
    L, M, spin = case["lmax"], case["mmax"], what.startswith("spin")
    flat = x.reshape(-1, x.shape[-1])
    if what == "round":
        maps = _exact_synth(flat, geom, L, M, False)
        return [maps, _exact_anal(maps, geom, L, M, False)]
    f = _exact_synth if what.endswith("synth") else _exact_anal
    got = f(flat, geom, L, M, spin)
    return got.reshape(x.shape[:-1] + got.shape[-1:])
