"""Device-resident Lanczos steps kept in flight: the explicit branch (a step
whose fused sums cancel) in the middle of enqueued chunks, runs shorter than a
chunk, and vectors stored for only part of a run."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _setup(lattice, nup, ndn, U):
    import paper_1204_3425_gb300 as hub
    from oracle.basis import Sector
    from workload import lattice_by_name
    ns, bonds = lattice_by_name(lattice)
    S = Sector(ns, bonds, nup, ndn, 1.0, U)
    return hub, hub.hubbard_sector_create(ns, bonds, nup, ndn, 1.0, U), S.explicit()


def _lanczos(Hx, v, m):
    f, old, a, b = v / np.linalg.norm(v), np.zeros_like(v), [], [0.0]
    for _ in range(m):
        w = Hx @ f - b[-1] * old
        a.append(f @ w)
        w -= a[-1] * f
        b.append(np.linalg.norm(w))
        f, old = w / b[-1], f
    return np.array(a), np.array(b[1:])


@pytest.mark.parametrize("lattice,nup,ndn,U", [("ring6", 3, 3, 4.0), ("ring8", 4, 3, 2.5), ("sq3x2", 2, 4, 8.0)])
@pytest.mark.parametrize("steps", [1, 2, 3, 5, 8, 9])
def test_explicit_branch_inside_the_pipeline(lattice, nup, ndn, U, steps):
    hub, H, Hx = _setup(lattice, nup, ndn, U)
    lam, Z = np.linalg.eigh(Hx.toarray())
    rng = np.random.default_rng(3)
    v = Z[:, 0] + 1e-5 * (rng.standard_normal(H.D) / np.sqrt(H.D))     # beta_2 ~ 1e-5: step 1 cancels
    r = hub.lanczos_ground_state(H, torch.from_numpy(v).cuda(), steps, 0.0)
    a, b = _lanczos(Hx, v, steps)
    # beta_2 carries an absolute error of some 1e-15 |H|, i.e. 1e-9 of itself here, which later steps inherit
    assert r["iters"] == steps
    assert np.allclose(r["alpha"], a, rtol=0, atol=1e-6 * np.abs(lam).max())
    assert np.allclose(r["beta"], b, rtol=0, atol=1e-6 * np.abs(lam).max())
    assert abs(r["alpha"][0] - a[0]) <= 1e-12 * abs(a[0])
    assert abs(r["beta"][0] - b[0]) <= 1e-8 * b[0]
    H.close()


@pytest.mark.parametrize("stored", [0, 1, 2, 5, 200])
def test_stored_vectors_end_inside_a_run(stored):
    hub, H, Hx = _setup("ring8", 4, 4, 4.0)
    E0 = np.linalg.eigvalsh(Hx.toarray())[0]
    v = torch.from_numpy(np.random.default_rng(5).uniform(-1, 1, H.D)).cuda()
    psi = torch.empty_like(v)
    r = hub.lanczos_ground_state_refined(H, v, 500, 1e-10, psi_out=psi, store_vectors=stored)
    assert abs(r["energy"] - E0) <= 1e-9 * abs(E0)
    p = psi.cpu().numpy()
    assert abs(p @ (Hx @ p) - E0) <= 1e-6 * abs(E0)
    H.close()


@pytest.mark.parametrize("lattice,nup,ndn,U,dtype", [("ring6", 1, 1, 4.0, "f64"), ("ring8", 4, 4, 7.3, "f32"),
                                                     ("ring13", 6, 6, 8.0, "f64"), ("ring13", 6, 7, 8.0, "f32")])
def test_ritz_vector_of_kept_and_replayed_vectors(lattice, nup, ndn, U, dtype):
    """All Lanczos vectors kept, or (2.9e6 elements: 46 of some 60 binary64 ones) the
    last part replayed: psi solves the eigenproblem to the residual reported, plus
    rounding (binary32: 2^-24 per element and operation, 1e-5 here)."""
    import paper_1204_3425_gb300 as hub
    from workload import lattice_by_name
    ns, bonds = lattice_by_name(lattice)
    H = hub.hubbard_sector_create(ns, bonds, nup, ndn, 1.0, U)
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    v = torch.rand(H.D, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    tol = 1e-9 if dtype == "f64" else 1e-4
    psi = torch.empty_like(v)
    r = hub.lanczos_ground_state(H, v if dtype == "f64" else v.float(), 400, tol, psi_out=psi)
    w = torch.empty_like(psi)
    hub.hubbard_apply(H, psi, w)
    theta = float(psi @ w)
    assert abs(float(psi.norm()) - 1.0) <= 1e-12
    assert abs(theta - r["energy"]) <= (1e-10 if dtype == "f64" else 1e-5) * abs(theta)
    assert float((w - theta * psi).norm()) <= 2 * tol + (1e-10 if dtype == "f64" else 1e-3)
    H.close()
