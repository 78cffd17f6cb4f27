"""The scalars of a Lanczos run, bit for bit.

The sums of a step are over the elements in one order, which the division of the
up phase's work over the threads fixes.  A run makes much of rounding (the step
it stops at, the late a_j and b_j, which nearby Ritz vector it mixes in, the sign
of psi), so another order is another result to a caller who compares runs.  The
golden values were recorded by `python -m tests.test_gpu_lanczos_bits` on a part of
152 SMs, with the order in use since the fused reductions came; the number of
SMs is part of it."""
import hashlib
import json
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "lanczos_bits.json")

# lattice, N_up, N_dn, U, dtype, steps (0: to a residual of 1e-10)
CASES = [
    ("ring6", 1, 1, 4.0, "f64", 0),        # one item, one column chunk
    ("sq3x3", 4, 4, 4.0, "f64", 0),        # fewer items than SMs
    ("ring7", 3, 3, 5.3, "f64", 0),        # and rows of odd length, the 128-bit epilogue
    ("ring12", 6, 6, 5.3, "f64", 0),       # several items a CTA
    ("ring12", 2, 5, 8.0, "f64", 0),       # about as many items as CTAs
    ("ring13", 5, 5, 2.0, "f64", 30),      # odd rows
    ("ring13", 6, 6, 8.0, "f64", 30),      # more than 2.5e6 elements
    ("ring13", 6, 6, 7.3, "f64", 60),      # the same; 45 vectors kept for psi, 15 replayed
    ("ring15", 5, 6, 7.3, "f64", 12),      # more than 2.5e6 elements, odd rows
    ("ring18", 2, 9, 7.3, "f64", 12),      # rows staged one word at a time
    ("ring16", 1, 8, 4.0, "f64", 0),       # 16 rows of 12870 elements
    ("ring10", 3, 0, 4.0, "f64", 0),       # one column
    ("ring14", 7, 7, 4.0, "f32", 40),      # binary32, 4 columns a lane
    ("ring13", 4, 3, 2.5, "f32", 40),      # 2
    ("ring13", 5, 4, 2.5, "f32", 40),      # 1
    ("sq3x3", 4, 4, 8.0, "f32", 40),
    ("ring16", 7, 7, 1.0, "f32", 8),       # 1.3e8 elements
]


def _run(lattice, nup, ndn, U, dtype, steps):
    import paper_1204_3425_gb300 as hub
    from workload import lattice_by_name, start_vector
    ns, bonds = lattice_by_name(lattice)
    H = hub.hubbard_sector_create(ns, bonds, nup, ndn, 1.0, U)
    v = torch.from_numpy(start_vector(H.D, seed=31)).cuda()
    v = v if dtype == "f64" else v.float()
    psi = torch.empty(H.D, dtype=torch.float64, device="cuda") if dtype == "f64" else None
    r = hub.lanczos_ground_state(H, v, steps or 1000, 0.0 if steps else 1e-10, psi_out=psi)
    H.close()
    ab = np.concatenate([r["alpha"], r["beta"]]) + 0.0
    out = dict(iters=r["iters"], energy=float(r["energy"]).hex(), last=[float(r["alpha"][-1]).hex(), float(r["beta"][-1]).hex()],
               scalars=hashlib.sha256(ab.tobytes()).hexdigest())
    if psi is not None:
        out["psi"] = hashlib.sha256((psi.cpu().numpy() + 0.0).tobytes()).hexdigest()
    return out


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%s-%d-%d-%g-%s" % c[:5])
def test_lanczos_scalars_are_the_recorded_ones(case):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("recorded on 152 SMs")
    with open(GOLDEN) as f:
        want = json.load(f)["%s-%d-%d-%g-%s" % case[:5]]
    assert _run(*case) == want


# binary32 vectors combined in binary64: lattice, N_up, N_dn, U
PSI_CASES = [("sq3x3", 4, 4, 4.0), ("ring11", 5, 6, 7.3), ("ring12", 6, 6, 4.0),
             ("ring14", 7, 7, 4.0)]      # 22 vectors of the plain run kept for psi, 38 replayed


def _psi32(lattice, nup, ndn, U, store):
    """The Ritz vector of the refined solver (store: vectors it may keep), or of a
    binary32 run (store None)."""
    import paper_1204_3425_gb300 as hub
    from workload import lattice_by_name, start_vector
    ns, bonds = lattice_by_name(lattice)
    H = hub.hubbard_sector_create(ns, bonds, nup, ndn, 1.0, U)
    v = torch.from_numpy(start_vector(H.D, seed=31)).cuda()
    psi = torch.empty_like(v)
    if store is None:
        r = hub.lanczos_ground_state(H, v.float(), 60, 0.0, psi_out=psi)
    else:
        r = hub.lanczos_ground_state_refined(H, v, 1000, 1e-10, psi_out=psi, store_vectors=store)
    H.close()
    return dict(energy=float(r["energy"]).hex(), psi=hashlib.sha256((psi.cpu().numpy() + 0.0).tobytes()).hexdigest())


@pytest.mark.parametrize("case", PSI_CASES, ids=lambda c: "%s-%d-%d-%g" % c)
def test_ritz_vectors_of_binary32_runs_are_the_recorded_ones(case):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("recorded on 152 SMs")
    with open(GOLDEN) as f:
        want = json.load(f)["psi32-%s-%d-%d-%g" % case]
    assert _psi32(*case, None) == want["run"]
    for store in (0, 1, 2, 9, 300):
        assert _psi32(*case, store) == want["refined"], store


def test_replayed_steps_sum_long_hop_lists_in_the_steps_order():
    """36 up-hops a state: more than a window of 32.  The replay's kernel stages its hop
    lists, the step's reads them; a psi of kept and of replayed vectors is the same."""
    import paper_1204_3425_gb300 as hub
    from workload import start_vector
    H = hub.hubbard_sector_create(10, [(i, j) for i in range(10) for j in range(i)], 6, 4, 1.0, 3.0)
    H2 = hub.hubbard_sector_create(12, [(i, j) for i in range(12) for j in range(i)], 6, 3, 1.0, 3.0)
    for h in (H, H2):
        v = torch.from_numpy(start_vector(h.D, seed=7)).cuda()
        psi = [torch.empty_like(v) for _ in range(3)]
        for p, store in zip(psi, (300, 0, 5)):
            hub.lanczos_ground_state_refined(h, v, 60, 1e-10, psi_out=p, store_vectors=store)
        assert torch.equal(psi[0], psi[1]) and torch.equal(psi[0], psi[2])
        h.close()


if __name__ == "__main__":
    got = {"%s-%d-%d-%g-%s" % c[:5]: _run(*c) for c in CASES}
    for c in PSI_CASES:
        got["psi32-%s-%d-%d-%g" % c] = dict(run=_psi32(*c, None), refined=_psi32(*c, 300))
    with open(GOLDEN, "w") as f:
        json.dump(got, f, indent=0)
        f.write("\n")
