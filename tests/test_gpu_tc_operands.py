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
