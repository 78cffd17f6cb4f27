"""Rounding of the binary64 H*v: with inputs on the fixed-point grid and integer
t, U the exact product is known as an integer, and the result is that integer
rounded once to binary64 (ties to even), whatever kernel forms it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("lattice,nup,ndn,U", [("ring8", 4, 4, 4), ("ring8", 3, 5, 0), ("sq3x3", 4, 5, 8),
                                               ("ring11", 4, 5, 1), ("ring11", 5, 4, 12), ("ring6", 1, 1, 2)])
@pytest.mark.parametrize("bits", [48, 30, 3])
def test_exact_products_round_once(lattice, nup, ndn, U, bits):
    import paper_1204_3425_gb300 as hub
    from oracle.basis import Sector
    from workload import lattice_by_name
    ns, bonds = lattice_by_name(lattice)
    S = Sector(ns, bonds, nup, ndn, 1.0, float(U))
    Hx = S.explicit().tocsr()
    rng = np.random.default_rng(ns * 100 + nup * 10 + bits)
    X = rng.integers(-(1 << bits) + 1, 1 << bits, size=S.D, dtype=np.int64)
    X[0] = (1 << 48) - 1                               # max|v| just below 1: the grid is 2^-48
    v = torch.from_numpy(X.astype(np.float64) * 2.0 ** -48).cuda()
    w = torch.empty_like(v)
    H = hub.hubbard_sector_create(ns, bonds, nup, ndn, 1.0, float(U))
    hub.hubbard_apply(H, v, w)
    got = w.cpu().numpy()
    coef = Hx.data.astype(np.int64)
    assert np.array_equal(coef, Hx.data)
    Xo = X.astype(object)
    want = np.empty(S.D)
    for r in range(S.D):
        sl = slice(Hx.indptr[r], Hx.indptr[r + 1])
        want[r] = float(sum(int(c) * int(x) for c, x in zip(coef[sl], Xo[Hx.indices[sl]]))) * 2.0 ** -48
    assert np.array_equal(got, want)
    H.close()


@pytest.mark.parametrize("nup,ndn,U", [(0, 8, 4.0), (1, 9, 7.3), (1, 10, 4.0), (2, 8, 0.0)])
def test_long_rows_match_the_reference_kernel(nup, ndn, U):
    """Rows of 43758 and 48620 elements: one word per element staged at a time.
    Bound: 1e-12 |t| max|v| for the fixed-point path plus the native kernel's own
    rounding, (W + U n) 2^-52 max|v| < 1e-13."""
    import paper_1204_3425_gb300 as hub
    from workload import ring
    H = hub.hubbard_sector_create(18, ring(18), nup, ndn, 1.0, U)
    v = torch.from_numpy(np.random.default_rng(7).uniform(-1, 1, H.D)).cuda()
    w, r = torch.empty_like(v), torch.empty_like(v)
    hub.hubbard_apply(H, v, w)
    hub.hubbard_apply_reference(H, v, r)
    assert float((w - r).abs().max()) <= 1.1e-12
    # the Lanczos step reads the same row sums: a_1, b_2 of a unit vector
    f = v / v.norm()
    res = hub.lanczos_ground_state(H, f, 3, 0.0)
    hub.hubbard_apply_reference(H, f, r)
    a = float(f @ r)
    b = float((r - a * f).norm())
    assert abs(res["alpha"][0] - a) <= 1e-11 * max(1.0, abs(a)) and abs(res["beta"][0] - b) <= 1e-11 * b
    H.close()


@pytest.mark.parametrize("lattice,nup,ndn,U", [
    ("sq4x4", 8, 3, 8.0),      # many rows, several column groups per row range
    ("sq4x4", 3, 8, 7.3),      # few rows, many chunks
    ("ring16", 8, 2, 4.0),     # short even rows
    ("ring16", 1, 8, 4.0),     # 16 rows
    ("ring13", 6, 5, 2.5),     # odd rows
    ("ring20", 10, 1, 4.0),    # more rows per range than lists fit at a time
    ("ring11", 5, 10, 4.0),    # a few columns
])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_up_phase_forms_match_the_reference_kernel(lattice, nup, ndn, U, dtype):
    """Every form of the up phase against one thread per element.  binary64: 1e-12
    max|v| plus the native kernel's rounding; binary32: 2^-24 per operation on
    either side, 2 (W + 2) 2^-24 max(1, U N) with W <= 48."""
    import paper_1204_3425_gb300 as hub
    from workload import lattice_by_name
    ns, bonds = lattice_by_name(lattice)
    H = hub.hubbard_sector_create(ns, bonds, nup, ndn, 1.0, U)
    g = torch.Generator(device="cuda")
    g.manual_seed(13)
    v = torch.rand(H.D, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    if dtype == "f32":
        v = v.float()
    w, r = torch.empty_like(v), torch.empty_like(v)
    hub.hubbard_apply_reference(H, v, r)
    bound = 1.2e-12 if dtype == "f64" else 2 * 50 * 2.0 ** -24 * max(1.0, U * min(nup, ndn))
    for _ in range(2):                                  # the second product reads an exponent word set back by the first
        w.fill_(float("nan"))
        hub.hubbard_apply(H, v, w)
        assert float((w - r).abs().max()) <= bound
    small = v * 2.0 ** -20                              # a smaller exponent must not meet the last one's
    hub.hubbard_apply(H, small, w)
    assert float((w * 2.0 ** 20 - r).abs().max()) <= bound
    H.close()
