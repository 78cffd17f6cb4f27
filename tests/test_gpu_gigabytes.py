"""binary32 products of vectors of more than 2 GiB, whose up phase has a kernel of its
own."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def sector():
    import paper_1204_3425_gb300 as hub
    from workload import ring
    H = hub.hubbard_sector_create(18, ring(18), 6, 7, 1.0, 4.0)     # 18564 x 31824: neither a multiple of its tile
    assert H.D * 4 > 2 << 30
    yield hub, H
    H.close()


def test_product_matches_the_reference_kernel(sector):
    """2^-24 for each of up to 26 hops and 2 more operations, on either side, of terms of
    at most max(1, U N) max|v|."""
    hub, H = sector
    g = torch.Generator(device="cuda")
    g.manual_seed(19)
    v = torch.rand(H.D, dtype=torch.float32, device="cuda", generator=g) * 2 - 1
    w, r = torch.full_like(v, float("nan")), torch.empty_like(v)
    hub.hubbard_apply(H, v, w)
    hub.hubbard_apply_reference(H, v, r)
    assert float(w.sub_(r).abs_().max()) <= 2 * 28 * 2.0 ** -24 * 4.0 * 6


def test_replayed_steps_are_the_stored_ones(sector):
    hub, H = sector
    g = torch.Generator(device="cuda")
    g.manual_seed(20)
    v = torch.rand(H.D, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    psi = [torch.empty_like(v) for _ in range(2)]
    for p, store in zip(psi, (8, 0)):                   # a bound that needs no polish
        hub.lanczos_ground_state_refined(H, v, 6, 1e6, psi_out=p, store_vectors=store)
    assert torch.equal(psi[0], psi[1])
