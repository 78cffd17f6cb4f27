"""Sectors with one spin empty or full: one row of any length.  Product and Lanczos
step against the one-thread-per-element kernel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("ns,nup,ndn,cols", [(22, 0, 6, 0), (22, 22, 6, 0), (22, 6, 0, 0), (23, 0, 7, 0), (24, 0, 12, 0),
                                             (18, 0, 9, 1), (18, 18, 9, 0), (25, 0, 11, 0), (8, 0, 0, 0)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_one_row_sectors(ns, nup, ndn, cols, dtype):
    """binary64: 1e-12 max|v| for the fixed point plus the native kernel's rounding, and
    the step's scalars to 1e-11 (the bounds of the long rows); binary32: 2^-24 for each
    of up to 24 hops and 2 more operations on either side, and the same for the scalars
    (sums of up to 4.5e6 products whose errors are not all of one sign)."""
    import paper_1204_3425_gb300 as hub
    from workload import ring
    H = hub.hubbard_sector_create(ns, ring(ns), nup, ndn, 1.0, 4.0)
    if cols:
        hub.hubbard_set_schedule(H, 0, cols, 0, 0)
    v = torch.from_numpy(np.random.default_rng(5).uniform(-1, 1, H.D)).cuda()
    v = v / v.norm() if H.D > 1 else v
    v = v if dtype == "f64" else v.float()
    scale = float(v.abs().max())
    eps = 1.1e-12 if dtype == "f64" else 2 * 26 * 2.0 ** -24 * max(1.0, 4.0 * min(nup, ndn))
    w, r = torch.empty_like(v), torch.empty_like(v)
    hub.hubbard_apply(H, v, w)
    hub.hubbard_apply_reference(H, v, r)
    assert float((w - r).abs().max()) <= eps * scale
    if dtype == "f32" and ndn and H.D > 50000:          # no binary32 step on rows longer than shared memory
        H.close()
        return
    res = hub.lanczos_ground_state(H, v, min(3, H.D), 0.0)
    f, r = v.double(), r.double()
    f = f / f.norm() if H.D > 1 else torch.ones_like(f)
    r = r if H.D > 1 else r / v.double()
    tol = 1e-11 if dtype == "f64" else eps
    a = float(f @ r)
    b = float((r - a * f).norm())
    assert abs(res["alpha"][0] - a) <= tol * max(1.0, abs(a))
    assert abs(res["beta"][0] - b) <= tol * max(b, 1.0)
    if H.D > 1:                                         # a step on the caller's vectors
        g = torch.zeros_like(v)
        a1, b2 = hub.hubbard_lanczos_step(H, v, g, 0.0)
        assert abs(a1 - a) <= tol * max(1.0, abs(a)) and abs(b2 - b) <= tol * max(b, 1.0)
        assert float((g.double() - (r - a * f) / b).abs().max()) <= 8 * tol * max(1.0, 1.0 / b)
    H.close()
