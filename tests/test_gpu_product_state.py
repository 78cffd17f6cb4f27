"""What a product leaves behind on its handle: nothing that another product, a replay
of a captured one or a Lanczos run on another stream can meet."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

# exponent found by the row phase; by a pass of its own (even rows, odd rows, long
# rows, more than 2.5e6 elements); by one word that a memset sets back
SECTORS = [("ring8", 4, 4), ("sq3x3", 4, 5), ("ring12", 6, 6), ("ring13", 6, 5), ("ring18", 1, 9), ("sq4x4", 5, 5),
           ("ring15", 7, 5), ("ring18", 3, 8)]


def _sector(lattice, nup, ndn, U=4.0):
    import paper_1204_3425_gb300 as hub
    from workload import lattice_by_name
    ns, bonds = lattice_by_name(lattice)
    return hub, hub.hubbard_sector_create(ns, bonds, nup, ndn, 1.0, U)


@pytest.mark.parametrize("lattice,nup,ndn", SECTORS)
def test_each_product_finds_its_own_exponent(lattice, nup, ndn):
    """w(2^k v) = 2^k w(v) to the last bit, in any order of the sizes: the grid follows
    the largest exponent of this product's vector alone."""
    hub, H = _sector(lattice, nup, ndn)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    v = torch.rand(H.D, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    want, w = torch.empty_like(v), torch.empty_like(v)
    hub.hubbard_apply(H, v, want)
    for k in (-30, 40, -900, 0, 0, 300, -1):
        x = v * 2.0 ** k
        w.fill_(float("nan"))
        hub.hubbard_apply(H, x, w)
        assert torch.equal(w, want * 2.0 ** k), k
    H.close()


@pytest.mark.parametrize("lattice,nup,ndn", SECTORS)
def test_captured_products_replay_on_new_values(lattice, nup, ndn):
    hub, H = _sector(lattice, nup, ndn)
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    v = torch.rand(H.D, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    want, w, x = torch.empty_like(v), torch.empty_like(v), v.clone()
    hub.hubbard_apply(H, v, want)                       # scratch allocated, kernel attributes set
    torch.cuda.synchronize()
    G = torch.cuda.CUDAGraph()
    with torch.cuda.graph(G):
        hub.hubbard_apply(H, x, w, stream=torch.cuda.current_stream())
        hub.hubbard_apply(H, x, w, stream=torch.cuda.current_stream())
    for k in (20, -20, 0):
        x.copy_(v * 2.0 ** k)
        w.fill_(float("nan"))
        G.replay()
        assert torch.equal(w, want * 2.0 ** k), k
    hub.hubbard_apply(H, v, w)
    assert torch.equal(w, want)
    del G
    H.close()


@pytest.mark.parametrize("lattice,nup,ndn", [("ring12", 6, 6), ("ring13", 6, 5), ("sq3x3", 4, 4), ("ring18", 1, 9)])
def test_run_beside_products_of_the_same_handle(lattice, nup, ndn):
    """Products still running on one stream when a run with a workspace of its own starts
    on another: both as if alone."""
    hub, H = _sector(lattice, nup, ndn, 5.3)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    v = torch.rand(H.D, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    f = torch.rand(H.D, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    want, w = torch.empty_like(v), torch.empty_like(v)
    ws = torch.empty(hub.lanczos_workspace_bytes(H), dtype=torch.uint8, device="cuda")
    hub.hubbard_apply(H, v, want)
    alone = hub.lanczos_ground_state(H, f, 40, 0.0, workspace=ws)
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(3):
        w.fill_(float("nan"))
        torch.cuda.synchronize()
        for _ in range(200):
            hub.hubbard_apply(H, v, w, stream=s1)
        r = hub.lanczos_ground_state(H, f, 40, 0.0, workspace=ws, stream=s2)
        torch.cuda.synchronize()
        assert np.array_equal(r["alpha"], alone["alpha"]) and np.array_equal(r["beta"], alone["beta"])
        assert torch.equal(w, want)
    H.close()
