"""Plans that find no device memory for the tables of the tensor-core kernels (injected on the host:
sht_debug_fail_allocations_after) run their Legendre steps, scalar and spin, on the plain FP64 kernels, as
every plan could before those tables were held."""
import numpy as np
import pytest

import oracle
from paper_1106_0159_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-11  # the FP64 bar of the parity tests


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def rel(x, ref):
    x, ref = x.cpu().numpy(), ref.cpu().numpy()
    return float(np.max(np.abs(x - ref)) / np.sqrt(np.mean(np.abs(ref) ** 2)))


def test_plans_without_memory_for_the_tensor_core_tables():
    from paper_1106_0159_gb300 import sht
    inject = sht.load().sht_debug_fail_allocations_after
    geom, L = sht.healpix_geometry(100), 200
    w = sht.Plan(geom, L)
    a = dev(inputs.gaussian_alm(L, L, seed=2, nmaps=2))
    e = dev(np.stack([inputs.gaussian_alm(L, L, seed=3, nmaps=2), inputs.gaussian_alm(L, L, seed=4, nmaps=2)], axis=1))
    m, s = w.alm2map(a), w.alm2map_spin(e)
    b, t = w.map2alm(m), w.map2alm_spin(s)
    torch.cuda.synchronize()
    plans, k = [], 0
    while len(plans) < 4:  # three tables: three failure points, then none
        inject(k)
        try:
            plans.append(sht.Plan(geom, L))
        except sht.ShtError as err:
            assert err.status == sht.SHT_ENOMEM and not plans, k
        finally:
            inject(-1)
        k += 1
        assert k < 100
    for p in plans[:3]:
        got = p.alm2map(a)
        assert not torch.equal(got, m) and rel(got, m) < TOL
        assert rel(p.map2alm(m), b) < TOL
        assert rel(p.alm2map_noalloc(a), m) < TOL
        assert p.workspace_bytes(2) > 0
    assert torch.equal(plans[3].alm2map(a), m) and torch.equal(plans[3].map2alm(m), b)
    # spin: two plain tables, whose failures stay ENOMEM, then the three of the tensor-core kernels
    p = plans[3]
    k = 0
    while True:
        inject(k)
        try:
            got = p.alm2map_spin(e)
            break
        except sht.ShtError as err:
            assert err.status == sht.SHT_ENOMEM
        finally:
            inject(-1)
        k += 1
        assert k < 100
    assert k >= 2 and not torch.equal(got, s) and rel(got, s) < TOL
    assert rel(p.map2alm_spin(s), t) < TOL
    assert torch.equal(p.alm2map_spin(e), got)   # and stays there
    # a batch of one such plan and one with its tables
    q = plans[0]
    o1, o2 = torch.zeros_like(m), torch.zeros_like(m)
    batch = sht.Batch(sht.BATCH_ALM2MAP, [(q, a, o1), (w, a, o2)])
    batch.run()
    torch.cuda.synchronize()
    assert torch.equal(o2, m) and torch.equal(o1, q.alm2map(a))
    batch.close()
    q.set_mode(sht.MODE_SPLIT_BF16)               # builds the tables now
    assert rel(q.alm2map(a), m) < 1e-9
