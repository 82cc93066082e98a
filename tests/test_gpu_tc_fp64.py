"""The Legendre steps of FP64 plans on the tensor cores (band limits from 192 on), scalar and spin 2: against
the oracle at the edges of their tiles (128-slot blocks, 32-l chunks, 4 / 8 / 16 maps), independent of how
maps are grouped, equal through every entry point, and with the plain kernels' results for values that
digits cannot carry.  Bars: max |x - oracle| / RMS <= 1e-11, the FP64 bar of the other parity tests;
equality bit for bit where the same sums run (class sums are exact integers)."""
import numpy as np
import pytest

import oracle
from oracle import geometry
from paper_1106_0159_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-11


def _plan(geom, L, M=None):
    from paper_1106_0159_gb300 import sht
    return sht.Plan(geom, L, M)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def rel(x, ref):
    x, ref = np.asarray(x), np.asarray(ref)
    return float(np.max(np.abs(x - ref)) / np.sqrt(np.mean(np.abs(ref) ** 2)))


def rings(n, seed=1, nphi=24):
    """n unpaired rings over both hemispheres, poles included: n slots, a geometry of no grid."""
    rng = np.random.default_rng(seed)
    th = np.sort(np.concatenate([[0.0, np.pi], rng.uniform(1e-3, np.pi - 1e-3, n - 2)]))
    return np.full(n, nphi, np.int64), th, rng.uniform(0, 6, n), rng.uniform(0.5, 2.0, n) / n


# slots 1 block less one, full, one over; l ranges of a chunk edge (l - m + 1 = 32 k, +- 1); mmax < lmax; the
# last two have enough blocks for the synthesis form of two CTAs per SM
@pytest.mark.parametrize("n,L,M,nmaps", [(127, 192, 192, 1), (128, 223, 31, 4), (129, 224, 192, 5),
                                         (257, 222, 60, 9), (40, 255, 255, 16), (130, 193, 0, 17),
                                         (513, 197, 197, 1), (520, 200, 200, 7)])
def test_legendre_steps_against_oracle(n, L, M, nmaps):
    geom = rings(n, seed=n)
    p = _plan(geom, L, M)
    a = inputs.uniform_alm(L, M, seed=n, nmaps=nmaps)
    d = host(p.legendre_synth(dev(a)))
    x = inputs.random_delta(n, M, seed=n + 1, nmaps=nmaps)
    b = host(p.legendre_anal(dev(x)))
    ms = sorted({0, M // 2, M})
    for g in sorted({0, nmaps // 2, nmaps - 1}):
        assert rel(d[g], oracle.delta_synth(geom, a[g], L, M)) < TOL
        ref = oracle.legendre_anal(geom, x[g].T[ms].copy(), L, np.array(ms))
        got = np.concatenate([b[g][oracle.alm_index(L, m, m):oracle.alm_index(L, m, m) + L - m + 1] for m in ms])
        assert rel(got, np.concatenate(ref)) < TOL
    assert np.all(b[:, :L + 1].imag == 0.0)
    for g in (0, nmaps - 1):  # a map's result does not depend on the maps beside it
        assert np.array_equal(host(p.legendre_synth(dev(a[g:g + 1])))[0], d[g])
        assert np.array_equal(host(p.legendre_anal(dev(x[g:g + 1])))[0], b[g])
    assert p.device_status() == 0


def test_every_entry_point_gives_the_same():
    from paper_1106_0159_gb300 import sht
    L = 200
    p = _plan(sht.healpix_geometry(100), L)
    a = dev(inputs.gaussian_alm(L, L, seed=3, nmaps=3))
    m = p.alm2map(a)
    b = p.map2alm(m)
    assert torch.equal(p.alm2map_noalloc(a), m)
    assert torch.equal(p.alm2map_ws(a, p.scratch(3)), m) and torch.equal(p.map2alm_ws(m, p.scratch(3)), b)
    m2, b2 = torch.zeros_like(m), torch.zeros_like(b)
    small = _plan(sht.healpix_geometry(32), 64)   # a plan of the queue beside it
    sa = dev(inputs.gaussian_alm(64, 64, seed=4))
    sm = torch.zeros((1, small.npix), dtype=torch.float64, device="cuda")
    syn = sht.Batch(sht.BATCH_ALM2MAP, [(p, a, m2), (small, sa, sm)])
    ana = sht.Batch(sht.BATCH_MAP2ALM, [(p, m, b2)])
    syn.run()
    ana.run()
    torch.cuda.synchronize()
    assert torch.equal(m2, m) and torch.equal(b2, b) and torch.equal(sm, small.alm2map(sa))
    syn.close()
    ana.close()
    ms = [0, 7, 199]
    full, back = host(p.legendre_synth(a)), host(b)
    p.set_mlist(ms)
    part = host(p.legendre_synth(a))
    bl = host(p.map2alm(m))
    mv = inputs.lm_arrays(L, L)[1]
    assert np.array_equal(part[:, :, ms], full[:, :, ms]) and not np.delete(part, ms, axis=2).any()
    assert np.array_equal(bl[:, np.isin(mv, ms)], back[:, np.isin(mv, ms)]) and not bl[:, ~np.isin(mv, ms)].any()


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e-310, 1e305])
def test_values_that_digits_cannot_carry(bad):
    """One such coefficient (or ring sum) in one map: its column is what the plain sums give, every other
    column and map keeps its bits."""
    L, n = 192, 60
    geom = rings(n, seed=9)
    p = _plan(geom, L)
    a = inputs.uniform_alm(L, L, seed=10, nmaps=3)
    d = host(p.legendre_synth(dev(a)))
    m = 5
    i = oracle.alm_index(L, m + 40, m)
    a[1, i] = bad
    e = host(p.legendre_synth(dev(a)))
    keep = np.ones(d.shape, bool)
    keep[1, :, m] = False
    assert np.array_equal(e[keep], d[keep])
    if np.isfinite(bad):
        big = max(1.0, abs(bad))
        assert rel(e[1, :, m] / big, oracle.delta_synth(geom, a[1], L, L)[:, m] / big) < TOL
    else:  # lambda is nonzero on every ring but the poles, whose dropped values still meet the coefficient
        assert not np.isfinite(e[1, 5:-5, m].real).any()
    x = inputs.random_delta(n, L, seed=11, nmaps=2)
    b = host(p.legendre_anal(dev(x)))
    x[1, n // 2, m] = bad
    c = host(p.legendre_anal(dev(x)))
    keep = np.ones(b.shape, bool)
    lo = oracle.alm_index(L, m, m)
    keep[1, lo:lo + L - m + 1] = False
    assert np.array_equal(c[keep], b[keep])
    if np.isfinite(bad):
        ref = oracle.legendre_anal(geom, x[1].T[[m]].copy(), L, np.array([m]))
        assert rel(c[1, lo:lo + L - m + 1] / big, np.concatenate(ref) / big) < TOL
    else:
        assert not np.isfinite(c[1, lo + 20:lo + L - m + 1].real).any()


@pytest.mark.parametrize("n,L,M,nmaps", [(97, 194, 194, 1), (200, 225, 40, 3), (193, 192, 2, 9)])
def test_spin_transforms_against_oracle(n, L, M, nmaps):
    geom = geometry.gauss_legendre(n, 2 * M + 3)
    p = _plan(geom, L, M)
    lv = inputs.lm_arrays(L, M)[0]
    a = np.stack([inputs.uniform_alm(L, M, seed=70 + n, nmaps=nmaps), inputs.uniform_alm(L, M, seed=80 + n, nmaps=nmaps)],
                 axis=1)
    s = host(p.alm2map_spin(dev(a)))          # l < 2 is ignored
    a[:, :, lv < 2] = 0.0
    rr = sorted({0, 1, n // 3, n // 2, n - 1})
    off = geometry.ring_offsets(geom)
    w = inputs.white_map(2 * geometry.npix(geom), seed=90 + n, nmaps=nmaps).reshape(nmaps, 2, -1)
    b = host(p.map2alm_spin(dev(w)))
    ms = sorted({0, 1, 2, M // 2, M})
    for g in sorted({0, nmaps - 1}):
        q, u = oracle.spin_alm2map_rings(geom, a[g, 0], a[g, 1], L, M, rr)
        got = [np.concatenate([s[g, k][off[r]:off[r + 1]] for r in rr]) for k in (0, 1)]
        assert rel(np.concatenate(got), np.concatenate([q, u])) < TOL
        Es, Bs = oracle.spin_map2alm_ms(geom, w[g, 0], w[g, 1], L, ms)
        sl = [slice(oracle.alm_index(L, m, m), oracle.alm_index(L, m, m) + L - m + 1) for m in ms]
        assert rel(np.concatenate([b[g, 0, k] for k in sl] + [b[g, 1, k] for k in sl]), np.concatenate(Es + Bs)) < TOL
        assert np.array_equal(host(p.alm2map_spin(dev(a[g:g + 1])))[0], s[g])
    assert not b[:, :, lv < 2].any() and not b[:, :, :L + 1].imag.any()
    if nmaps > 1:  # one map's E, B not finite: the other maps keep their bits
        a[0, 1, -1] = np.nan
        t = host(p.alm2map_spin(dev(a)))
        assert np.array_equal(t[1:], s[1:]) and np.isnan(t[0]).any()


# rings of direct prime radices (7 .. 113 and, above, those cheaper than Bluestein's form), of Bluestein
# primes, products, squares, and lengths shorter than the threads that share their folding
@pytest.mark.parametrize("smem", [1, 0])
@pytest.mark.parametrize("mode", [0, 1])
def test_ring_radices(smem, mode):
    from paper_1106_0159_gb300 import sht
    nphi = np.array([1, 2, 3, 4, 6, 9, 15, 19, 25, 4 * 23, 4 * 61, 8 * 89, 127, 4 * 131, 251, 257, 2 * 263, 521, 49 * 4,
                     3 * 5 * 7 * 11, 23 * 89, 4 * 509, 12 * 131], np.int64)
    n = len(nphi)
    rng = np.random.default_rng(8)
    geom = (nphi, np.sort(rng.uniform(0.05, 3.0, n)), rng.uniform(0, 6, n), rng.uniform(0.5, 2.0, n))
    M = 700
    p = _plan(geom, M, M)
    p.set_mode(mode)
    p.set_tuning(sht.TUNE_RING_SMEM, smem)
    d = inputs.random_delta(n, M, seed=12)
    s = inputs.white_map(geometry.npix(geom), seed=13)
    tol = TOL if mode == 0 else 1e-9
    assert rel(host(p.ring_synth(dev(d)))[0], oracle.ring_synth(geom, d[0], M)) < tol
    assert rel(host(p.ring_anal(dev(s)))[0], oracle.delta_anal(geom, s[0], np.arange(M + 1)).T) < tol
