"""A Lanczos step on the caller's vectors, element by element, in every form of its
kernels, against the one-thread-per-element product."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("lattice,nup,ndn,U", [
    ("ring6", 1, 1, 4.0),      # one item
    ("sq3x3", 4, 4, 4.0),      # fewer items than SMs, a row a warp
    ("ring7", 3, 3, 5.3),      # the same, odd rows
    ("ring11", 5, 9, 8.0),     # 55 columns, 28.9 items of 16 rows
    ("ring12", 6, 6, 5.3),     # several items a CTA
    ("ring13", 5, 5, 7.3),     # odd rows
    ("ring13", 6, 6, 8.0),     # more than 2.5e6 elements
    ("ring15", 6, 5, 2.0),     # the same, odd rows
    ("ring18", 1, 9, 7.3),     # 48620 columns: two words an element
    ("ring18", 3, 8, 4.0),     # 43758 columns, 816 rows: gathered from L2
    ("ring16", 0, 8, 4.0),     # one row
    ("ring16", 8, 0, 4.0),     # one column
])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_step_forms_match_the_reference_kernel(lattice, nup, ndn, U, dtype):
    """g <- (H f - beta g - a f) / b.  binary64: 1e-12 max|f| for the fixed point, as much
    for g on the same grid; binary32: 2^-24 for each of up to 50 operations on either
    side.  a and the norm are sums of all elements and far better than one element; a
    factor 3 covers them and the division."""
    import paper_1204_3425_gb300 as hub
    from workload import lattice_by_name
    ns, bonds = lattice_by_name(lattice)
    H = hub.hubbard_sector_create(ns, bonds, nup, ndn, 1.0, U)
    rnd = torch.Generator(device="cuda")
    rnd.manual_seed(17)
    f, g = (torch.rand(H.D, dtype=torch.float64, device="cuda", generator=rnd) * 2 - 1 for _ in range(2))
    f, g = f / f.norm(), g / g.norm()
    if dtype == "f32":
        f, g = f.float(), g.float()
    beta = 1.75
    r = torch.empty_like(f)
    hub.hubbard_apply_reference(H, f, r)
    w = torch.empty_like(f)
    hub.hubbard_apply(H, f, w)                          # and the product of the same sector
    eps = 2.4e-12 if dtype == "f64" else 2 * 50 * 2.0 ** -24 * max(1.0, U * min(nup, ndn))
    assert float((w.double() - r.double()).abs().max()) <= eps * float(f.abs().max())
    w = r.double() - beta * g.double()
    f64 = f.double()
    a = float(w @ f64)
    w -= a * f64
    b = float(w.norm())
    size = max(float(f.abs().max()), beta * float(g.abs().max()))
    a1, b2 = hub.hubbard_lanczos_step(H, f, g, beta)
    assert abs(a1 - a) <= eps * max(1.0, abs(a)) and abs(b2 - b) <= eps * max(1.0, b)
    assert float((g.double() - w / b).abs().max()) <= 3 * eps * size * max(1.0, 1.0 / b)
    H.close()
