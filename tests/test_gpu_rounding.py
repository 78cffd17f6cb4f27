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
