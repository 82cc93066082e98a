"""The largest call that sht_alm2map_noalloc takes: Delta and one ring buffer of 48 bytes per pixel of the
longest ring within sht_noalloc_scratch_bytes(), also where all rings are short."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_short_rings_up_to_the_documented_limit():
    from paper_1106_0159_gb300 import sht
    cap = int(sht.load().sht_noalloc_scratch_bytes())
    nphi, M = 16, 99
    per_map = 2 * (M + 1) * 16
    nmaps = cap // per_map
    left = cap - (nmaps * per_map + 255) // 256 * 256
    assert 48 * nphi <= left < 8192
    p = sht.Plan((np.full(2, nphi, np.int64), np.array([1.0, 2.0]), np.zeros(2), np.ones(2)), M)
    a = torch.randn(nmaps + 1, p.nalm, dtype=torch.float64, device="cuda").to(torch.complex128)
    got = p.alm2map_noalloc(a[:nmaps])
    assert torch.equal(got, p.alm2map(a[:nmaps]))
    with pytest.raises(ValueError):
        p.alm2map_noalloc(a)
    p.close()
