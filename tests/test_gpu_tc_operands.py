"""The tensor-core Legendre steps on operands that are not random draws: coefficients whose digits agree with
those of the recurrence, coefficients that run into the subnormal range, and m lists."""
import numpy as np
import pytest

import oracle
from paper_1106_0159_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _plan(geom, L, M=None):
    from paper_1106_0159_gb300 import sht
    return sht.Plan(geom, L, M)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


RINGS = (np.full(4, 16, np.int64), np.array([0.9, 1.2, 0.5 * np.pi, 1.9]), np.zeros(4), np.ones(4))


# On the equator y_l = -y_(l-2): with a_lm = S lambda_lm(pi/2) (a source there) or S sign(y) both operands of
# the sum over l repeat their digits, and the sums of digit products grow with the number of terms.  Bar:
# c_lm is a product of l / 2 factors of at most 3 roundings, 1.5 l 2^-53 at the end and half of it on
# average; the oracle's a_lm, in long double, gives the other half: 1.5 lmax 2^-53 of the largest sum.
@pytest.mark.parametrize("L,ms", [(4096, [0, 168, 288, 352]), (8191, [0]), (16383, [0])])
def test_coherent_operands(L, ms):
    M, nmaps = max(ms), 16
    p = _plan(RINGS, L, M)
    a = np.zeros((nmaps, oracle.nalm(L, M)), np.complex128)
    for m in ms:
        lam = oracle.lambda_lm(0.5 * np.pi, L, m)
        i = oracle.alm_index(L, m, m)
        for g in range(nmaps):
            S = 1.789903 * 2.0 ** (g / 16.0)
            a[g, i:i + L - m + 1] = S * lam + (1j * S * np.sign(lam) if m else 0.0)
    d = host(p.legendre_synth(dev(a)))
    for g in range(nmaps):
        ref = oracle.delta_synth(RINGS, a[g], L, M)
        for m in ms:
            for x, r in ((d[g, :, m].real, ref[:, m].real), (d[g, :, m].imag, ref[:, m].imag)):
                assert np.max(np.abs(x - r)) <= 1.5 * L * 2.0 ** -53 * max(np.max(np.abs(r)), 1e-300), (g, m)
    # the same bits in groups of 1 and 5 maps, and with enough CTAs for two per SM
    assert np.array_equal(host(p.legendre_synth(dev(a[:1])))[0], d[0])
    assert np.array_equal(host(p.legendre_synth(dev(a[3:8]))), d[3:8])
    assert p.device_status() == 0
    if L == 4096:
        W = 800
        w = np.zeros((1, oracle.nalm(L, W)), np.complex128)
        w[0, :a.shape[1]] = a[0]
        assert np.array_equal(host(_plan(RINGS, L, W).legendre_synth(dev(w)))[0, :, :M + 1], d[0])


def test_subnormal_values_beside_ordinary_ones():
    """Coefficients of a strongly smoothed spectrum pass through the subnormal range.  Beside a column's
    ordinary values they are below 2^-99 of its scale: the results are those with zeros there, bit for bit,
    which the plain sums are not."""
    L, n = 260, 140
    rng = np.random.default_rng(5)
    geom = (np.full(n, 8, np.int64), np.sort(rng.uniform(0.2, 2.9, n)), np.zeros(n), np.ones(n))
    p = _plan(geom, L)
    lv, mv = inputs.lm_arrays(L, L)
    a = inputs.uniform_alm(L, L, seed=6, nmaps=6) * np.exp(-0.5 * (lv * 0.15) ** 2)
    tiny = (np.abs(a.real) < 2.0 ** -1022) & (np.abs(a.imag) < 2.0 ** -1022)
    assert (tiny & (a != 0.0) & (mv < 200)).any(axis=1).all()
    z = np.where(tiny, 0.0, a)
    d, e = host(p.legendre_synth(dev(a))), host(p.legendre_synth(dev(z)))
    assert np.array_equal(d[:, :, :200], e[:, :, :200])
    t = inputs.uniform_alm(L, L, seed=8, nmaps=6).reshape(3, 2, -1)
    t[:, :, lv == 255] = 0.0
    w = host(p.alm2map_spin(dev(t)))
    t[:, :, (lv == 255) & (mv < 250)] = 1e-310 * (1.0 + 1j)
    assert np.array_equal(host(p.alm2map_spin(dev(t))), w)
    x = inputs.random_delta(n, L, seed=7, nmaps=6)
    x[:, ::7] = 0.0
    b = host(p.legendre_anal(dev(x)))
    x[:, ::7, 1:] = 3e-309 * (1.0 - 1j)
    assert np.array_equal(host(p.legendre_anal(dev(x))), b)
    assert p.device_status() == 0


@pytest.mark.parametrize("scale", [2.0 ** -950, 2.0 ** -1010, 2.0 ** -1030])
def test_columns_near_the_lower_end_of_the_range(scale):
    """Coefficients that are all tiny, some or all of them subnormal: the FP64 bar on Delta, plus for results
    below the normal range one rounding to a multiple of 2^-1074 and that of each input (the scaled
    oracle's inputs are the stored ones, so only the result's counts)."""
    L, M, n = 200, 30, 60
    rng = np.random.default_rng(15)
    geom = (np.full(n, 8, np.int64), np.sort(rng.uniform(0.2, 2.9, n)), np.zeros(n), np.ones(n))
    p = _plan(geom, L, M)
    a = inputs.uniform_alm(L, M, seed=16, nmaps=2) * scale
    d = host(p.legendre_synth(dev(a)))
    for g in (0, 1):
        ref = oracle.delta_synth(geom, a[g] * 2.0 ** 900, L, M)
        bar = 1e-11 * np.sqrt(np.mean(np.abs(ref) ** 2)) + 2.0 ** (900 - 1074)
        got = d[g] * 2.0 ** 900
        assert np.max(np.abs(got.real - ref.real)) <= bar and np.max(np.abs(got.imag - ref.imag)) <= bar


def test_an_m_list_cuts_the_coefficients_of_its_m_only():
    """A plan with an m list (one rank's share) reads and cuts no other m's coefficients: the rest of its scratch
    stays as it was."""
    L = 500
    p = _plan((np.full(8, 16, np.int64), np.linspace(0.4, 2.7, 8), np.zeros(8), np.ones(8)), L)
    a = dev(inputs.uniform_alm(L, L, seed=31))
    s = p.scratch(1)
    full = p.alm2map_ws(a, s).clone()
    p.set_mlist([0, 3])
    s.fill_(0xA5)
    got = p.alm2map_ws(a, s)
    assert float((s == 0xA5).double().mean()) > 0.9
    b = a.clone()
    b[:, oracle.alm_index(L, 4, 4):] = 0.0
    b[:, oracle.alm_index(L, 1, 1):oracle.alm_index(L, 3, 3)] = 0.0
    p.set_mlist()
    assert torch.equal(p.alm2map(b), got) and not torch.equal(got, full)


# Slots far below their block's scale, and what is bright on them.  The plain FP64 sums lose nothing to
# the other slots of a block; bar 1e-11, the FP64 bar of the parity tests, against each column's own RMS
# (analysis) and against each ring's own sum of |a_lm lambda_lm| (synthesis; above the dropping threshold).
SLOTS, BAND = 150, 256


def _slots_geom():
    th = np.concatenate([[0.025, 0.03], np.linspace(0.05, 0.5 * np.pi - 0.01, SLOTS - 2)])
    return np.full(SLOTS, 8, np.int64), th, np.zeros(SLOTS), np.ones(SLOTS)


@pytest.mark.parametrize("nmaps", [1, 7, 16])
def test_a_bright_polar_ring_leaves_the_other_columns_alone(nmaps):
    geom, ms = _slots_geom(), [0, 1, 20, 60, 150, 250]
    p = _plan(geom, BAND)
    x = inputs.random_delta(SLOTS, BAND, seed=41, nmaps=nmaps)
    x[:, 0] *= 1e9
    x[:, 1] *= 1e6
    b = host(p.legendre_anal(dev(x)))
    for g in {0, nmaps - 1}:
        ref = oracle.legendre_anal(geom, x[g].T[ms].copy(), BAND, np.array(ms))
        for m, r in zip(ms, ref):
            i = oracle.alm_index(BAND, m, m)
            assert np.max(np.abs(b[g, i:i + BAND - m + 1] - r)) <= 1e-11 * np.sqrt(np.mean(np.abs(r) ** 2)), (g, m)


@pytest.mark.parametrize("nmaps", [1, 16])
def test_every_ring_keeps_its_own_precision(nmaps):
    geom = _slots_geom()
    p = _plan(geom, BAND)
    a = inputs.uniform_alm(BAND, BAND, seed=43, nmaps=nmaps)
    d = host(p.legendre_synth(dev(a)))
    ref = oracle.delta_synth(geom, a[-1], BAND, BAND)
    seen = 0
    for m in (0, 5, 30, 80, 160, 250):
        i = oracle.alm_index(BAND, m, m)
        am = np.abs(a[-1, i:i + BAND - m + 1])
        for r in range(0, SLOTS, 3):
            tot = float(np.sum(am * np.abs(oracle.lambda_lm(float(geom[1][r]), BAND, m))))
            if tot > 1e-50:
                assert abs(d[-1, r, m] - ref[r, m]) <= 1e-11 * tot, (m, r)
                seen += tot < 1e-12
    assert seen > 10  # rings far below the others of their block


def test_a_batch_follows_its_plans_knobs():
    """The maps per launch set on a plan after the batch was made: the batch's own scratch serves both settings."""
    from paper_1106_0159_gb300 import sht
    p = _plan(RINGS, 400, 0)
    a = dev(inputs.uniform_alm(400, 0, seed=51, nmaps=12))
    want = p.alm2map(a)
    p.set_tuning(sht.TUNE_TC_MAPS, 8)
    out = torch.zeros_like(want)
    b = sht.Batch(sht.BATCH_ALM2MAP, [(p, a, out)])
    for maps in (16, 8):
        p.set_tuning(sht.TUNE_TC_MAPS, maps)
        out.zero_()
        b.run()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
    b.close()


# Grids without rings near the equator: there a column's terms can all lie far below the product of its
# scales (the largest coefficient at an l whose lambda is tiny on every ring).  Bar 1e-11 of the RMS of the
# map's Delta, resp. of the map, the FP64 bar of the parity tests.
def test_single_modes_on_a_polar_cap():
    n, L = 140, 300
    geom = (np.full(n, 8, np.int64), np.linspace(0.05, 0.9, n), np.zeros(n), np.ones(n))
    p = _plan(geom, L)
    modes = [(0, 0), (2, 2), (50, 50), (100, 100), (150, 150), (140, 100), (300, 260)]
    a = np.zeros((len(modes) + 1, oracle.nalm(L, L)), np.complex128)
    for g, (l, m) in enumerate(modes):
        a[g, oracle.alm_index(L, l, m)] = 0.7 + (0.4j if m else 0.0)
    a[-1] = inputs.uniform_alm(L, L, seed=61)[0]
    d = host(p.legendre_synth(dev(a)))
    for g in range(len(a)):
        ref = oracle.delta_synth(geom, a[g], L, L)
        assert np.max(np.abs(d[g] - ref)) <= 1e-11 * np.sqrt(np.mean(np.abs(ref) ** 2)), g
        assert np.array_equal(host(p.legendre_synth(dev(a[g:g + 1])))[0], d[g])
    p.set_mlist([100, 140])
    assert np.array_equal(host(p.legendre_synth(dev(a)))[3, :, 100], d[3, :, 100])


def test_steep_zonal_polarisation_near_the_pole():
    n, L = 30, 2000
    geom = (np.full(n, 16, np.int64), np.linspace(1e-4, 1e-3, n), np.zeros(n), np.ones(n))
    p = _plan(geom, L, 0)
    a = (inputs.uniform_alm(L, 0, seed=62, nmaps=2) * (1.0 + np.arange(L + 1)) ** -8.0)[None]
    s = host(p.alm2map_spin(dev(a)))
    q, u = oracle.spin_alm2map_rings(geom, a[0, 0], a[0, 1], L, 0, list(range(n)))
    ref, got = np.concatenate([q, u]), s[0].reshape(-1)
    assert np.max(np.abs(got - ref)) <= 1e-11 * np.sqrt(np.mean(ref ** 2))
