"""Performance cases: the work a user of the library has it do, each through
its public entry points.

A case is a sector (lattice, fillings, U) and an operation on it:
  apply    w = H v, binary64 or binary32 (hubbard_apply)
  lanczos  a fixed number of Lanczos steps (lanczos_ground_state, tol = 0):
           the time per iteration the paper quotes
  solve    a ground state to rho < 1e-10 with its Ritz vector
  refined  a ground state by the binary32 Lanczos with binary64 refinement, its
           Ritz vector kept at the accuracy it has (binary32)
  evolve   exp(-i H t) v of a complex v, Lanczos vectors stored
  batch    many uneven small sectors solved in one launch
Lattices are the rings and periodic rectangles of the workloads; U is a small
integer where a single sector is studied and any real in [0, 12] where it is
swept.
"""
import itertools
import math
import random

import numpy as np
import torch

import paper_1204_3425_gb300 as hub

MAX_ITERS = 1000
TOL = 1e-10
# Lanczos steps a run to TOL cannot do without, for work(): what uniform
# random start vectors take on these sectors is 60 to 160
SOLVE_STEPS = 80
EVOLVE_STEPS = 16

RINGS = ["ring%d" % n for n in range(6, 17)]
GRIDS = ["sq3x2", "sq4x2", "sq3x3", "sq4x3", "sq4x4"]
BATCH_LATTICES = ["ring%d" % n for n in range(6, 13)] + ["sq3x2", "sq4x2", "sq3x3", "sq4x3"]


def listed():
    return [
        # one product of a small ring: all launch and call latency (validation, teaching sizes)
        dict(name="apply_ring8_f64", op="apply", lattice="ring8", nup=4, ndn=4, U=4.0, dtype="f64"),
        # an ordinary half-filled sector: L2-resident vectors
        dict(name="apply_ring12_f64", op="apply", lattice="ring12", nup=6, ndn=6, U=4.0, dtype="f64"),
        # a doped ring with odd row length in binary32
        dict(name="apply_ring13_f32_odd", op="apply", lattice="ring13", nup=7, ndn=5, U=2.5, dtype="f32"),
        # rows of 48620 elements (one spin dilute, the other half-filled), U from a sweep
        dict(name="apply_ring18_f64_long_rows", op="apply", lattice="ring18", nup=2, ndn=9, U=7.3, dtype="f64"),
        # the paper's largest square lattice, both precisions: HBM-sized vectors
        dict(name="apply_sq4x4_f64", op="apply", lattice="sq4x4", nup=8, ndn=8, U=8.0, dtype="f64"),
        dict(name="apply_sq4x4_f32", op="apply", lattice="sq4x4", nup=8, ndn=8, U=8.0, dtype="f32"),
        # Lanczos iterations on the same sector
        dict(name="lanczos_sq4x4_f64", op="lanczos", lattice="sq4x4", nup=8, ndn=8, U=8.0, steps=8),
        # ground states one at a time: a small cluster, and an ordinary sector
        dict(name="solve_sq3x3_f64", op="solve", lattice="sq3x3", nup=4, ndn=4, U=4.0),
        dict(name="solve_ring12_f64", op="solve", lattice="ring12", nup=6, ndn=6, U=5.3),
        # a large sector by the mixed-precision route
        dict(name="refined_ring14", op="refined", lattice="ring14", nup=7, ndn=7, U=4.0),
        # time propagation of a complex state
        dict(name="evolve_sq4x3", op="evolve", lattice="sq4x3", nup=6, ndn=6, U=8.0, t=0.25),
        # a sweep over small sectors, as the batched workload draws them
        dict(name="batch_256", op="batch", count=256, list_seed=1234),
    ]


def draw(rng):
    op = rng.choice(["apply", "apply", "apply", "lanczos", "solve", "solve", "refined", "evolve", "batch"])
    if op == "batch":
        return dict(op=op, count=int(round(16 * 16 ** rng.random())), list_seed=rng.randrange(1 << 30))
    lo, hi = {"apply": (2e2, 1.66e8), "lanczos": (1e5, 1.66e8), "solve": (2e2, 9e5), "refined": (2e6, 1.2e7),
              "evolve": (2e2, 1.2e6)}[op]
    want = lo * (hi / lo) ** rng.random()
    sectors = [(lat, a, b) for lat in RINGS + GRIDS for a, b in itertools.product(range(1, _ns(lat)), repeat=2)
               if want / 1.5 <= _dim(lat, a, b) <= min(hi, want * 1.5)]
    lat, nup, ndn = rng.choice(sorted(sectors))
    case = dict(op=op, lattice=lat, nup=nup, ndn=ndn,
                U=float(rng.choice([1, 2, 4, 8])) if rng.random() < 0.5 else round(rng.uniform(0.0, 12.0), 3))
    if op == "apply":
        case["dtype"] = rng.choice(["f64", "f64", "f32"])
    if op == "lanczos":
        case["steps"] = rng.choice([4, 6, 8])
    if op == "evolve":
        case["t"] = round(rng.uniform(0.05, 0.3), 3)
    return case


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["op"] == "batch":
        specs = [(_ns(q["lattice"]), _bonds(q["lattice"]), q["nup"], q["ndn"], 1.0, q["U"]) for q in _batch_list(case)]
        B = hub.Batch(specs)
        v0 = torch.zeros(int(B.offsets[-1]), dtype=torch.float64, device=dev)
        for k, v in enumerate(_batch_starts(case, seed)):
            v0[int(B.offsets[k]):int(B.offsets[k]) + v.numel()] = v
        return dict(op="batch", B=B, v0=v0, ws=torch.empty(B.workspace_bytes(MAX_ITERS), dtype=torch.uint8, device=dev))
    H = hub.hubbard_sector_create(_ns(case["lattice"]), _bonds(case["lattice"]), case["nup"], case["ndn"], 1.0, case["U"])
    s = dict(op=case["op"], H=H)
    if case["op"] == "apply":
        s["v"] = _start(H.D, seed).to(torch.float64 if case["dtype"] == "f64" else torch.float32)
        s["w"] = torch.empty_like(s["v"])
    elif case["op"] == "evolve":
        re, im = _complex_start(H.D, seed)
        s.update(re=re, im=im, t=case["t"], out_re=torch.empty_like(re), out_im=torch.empty_like(im),
                 ws=torch.empty(hub.hubbard_evolve_workspace_bytes(H, 40), dtype=torch.uint8, device=dev))
    elif case["op"] == "refined":
        s["v"] = _start(H.D, seed)
        s["psi"] = torch.empty_like(s["v"])
        s["ws"] = torch.empty(hub.lanczos_refined_workspace_bytes(H, 128), dtype=torch.uint8, device=dev)
    else:
        s["v"] = _start(H.D, seed)
        s["ws"] = torch.empty(hub.lanczos_workspace_bytes(H), dtype=torch.uint8, device=dev)
        s["steps"] = case.get("steps")
        if case["op"] == "solve":
            s["psi"] = torch.empty_like(s["v"])
    return s


def run(state):
    op = state["op"]
    if op == "apply":
        return hub.hubbard_apply(state["H"], state["v"], state["w"])
    if op == "lanczos":
        r = hub.lanczos_ground_state(state["H"], state["v"], state["steps"], 0.0, workspace=state["ws"])
        return dict(energy=r["energy"], alpha=r["alpha"], beta=r["beta"])
    if op == "solve":
        r = hub.lanczos_ground_state(state["H"], state["v"], MAX_ITERS, TOL, workspace=state["ws"], psi_out=state["psi"])
        return dict(energy=r["energy"], psi=state["psi"])
    if op == "refined":
        r = hub.lanczos_ground_state_refined(state["H"], state["v"], MAX_ITERS, TOL, workspace=state["ws"],
                                             psi_out=state["psi"])
        return dict(energy=r["energy"], psi=state["psi"].float())
    if op == "evolve":
        re, im, _ = hub.hubbard_time_evolve(state["H"], state["re"], state["im"], state["t"], krylov_max=40, tol=TOL,
                                            workspace=state["ws"], out_re=state["out_re"], out_im=state["out_im"])
        return dict(re=re, im=im)
    state["B"].solve_async(state["v0"], MAX_ITERS, TOL, state["ws"])
    return np.array([r["energy"] for r in state["B"].results(state["ws"], MAX_ITERS)])


def work(case):
    """An H*v reads v and writes w and adds every hop; a Lanczos step reads f_j
    and f_{j-1} and writes f_{j+1}; a Ritz vector or a propagated state takes
    the vectors once more."""
    if case["op"] == "batch":
        parts = [work(dict(q, op="lanczos", steps=SOLVE_STEPS)) for q in _batch_list(case)]
        return dict(bytes=sum(p["bytes"] for p in parts), flops=sum(p["flops"] for p in parts))
    ns, D = _ns(case["lattice"]), _dim(case["lattice"], case["nup"], case["ndn"])
    nb = len(_bonds(case["lattice"]))
    hops = sum(2.0 * nb * math.comb(ns - 2, n - 1) / math.comb(ns, n) for n in (case["nup"], case["ndn"]))
    hv = D * (hops + 3.0)
    op, s = case["op"], 4 if case.get("dtype") == "f32" else 8
    if op == "apply":
        return dict(bytes=2.0 * D * s, flops=hv)
    m = min(D, {"lanczos": case.get("steps", 0), "evolve": 2 * EVOLVE_STEPS}.get(op, SOLVE_STEPS))
    size = 4 if op == "refined" else 8
    again = {"solve": 1.0, "refined": 1.0, "evolve": 1.0}.get(op, 0.0)
    return dict(bytes=m * D * size * (3.0 + again), flops=m * (hv + 6.0 * D + 2.0 * again * D))


def exact(case, seed):
    """What run() returns, by torch in binary64 from the definition of H."""
    op = case["op"]
    if op == "batch":
        return np.array([_ground(_Dense(q["lattice"], q["nup"], q["ndn"], q["U"]), v)[0]
                         for q, v in zip(_batch_list(case), _batch_starts(case, seed))])
    H = _Dense(case["lattice"], case["nup"], case["ndn"], case["U"])
    if op == "apply":
        v = _start(H.D, seed)
        return H(v.float().double() if case["dtype"] == "f32" else v)
    if op == "lanczos":
        a, b, _ = _krylov(H, _start(H.D, seed), case["steps"], keep=False)
        T = np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1)
        return dict(energy=float(np.linalg.eigvalsh(T)[0]), alpha=a, beta=b)
    if op == "evolve":
        re, im = _complex_start(H.D, seed)
        out = [torch.zeros_like(re), torch.zeros_like(re)]
        for part, mul in ((re, 1.0), (im, 1.0j)):
            a, b, F = _krylov(H, part, 60)
            lam, Z = np.linalg.eigh(np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1))
            y = mul * float(part.norm()) * (Z @ (np.exp(-1j * lam * case["t"]) * Z[0]))
            for k, c in enumerate((y.real, y.imag)):
                out[k] += torch.from_numpy(np.ascontiguousarray(c)).to(F) @ F[:len(a)]
        return dict(re=out[0], im=out[1])
    E, psi = _ground(H, _start(H.D, seed), vector=True)
    return dict(energy=E, psi=psi)


def _ns(lattice):
    if lattice.startswith("ring"):
        return int(lattice[4:])
    lx, ly = lattice[2:].split("x")
    return int(lx) * int(ly)


def _bonds(lattice):
    """Nearest neighbours of the ring, or of the periodic lx-by-ly rectangle (site x + lx y)."""
    if lattice.startswith("ring"):
        lx, ly = _ns(lattice), 1
    else:
        lx, ly = (int(a) for a in lattice[2:].split("x"))
    pairs = set()
    for y, x in itertools.product(range(ly), range(lx)):
        for j in ((x + 1) % lx + lx * y, x + lx * ((y + 1) % ly)):
            i = x + lx * y
            if i != j:
                pairs.add((min(i, j), max(i, j)))
    return sorted(pairs)


def _dim(lattice, nup, ndn):
    return math.comb(_ns(lattice), nup) * math.comb(_ns(lattice), ndn)


def _start(D, seed):
    """Random start vector, uniform in [-1, 1)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return 2.0 * torch.rand(D, dtype=torch.float64, device="cuda", generator=g) - 1.0


def _complex_start(D, seed):
    re, im = _start(D, 2 * int(seed)), _start(D, 2 * int(seed) + 1)
    n = float(torch.sqrt(re.square().sum() + im.square().sum()))
    return re / n, im / n


def _batch_list(case):
    r = random.Random(case["list_seed"])
    out = []
    for _ in range(case["count"]):
        lat = r.choice(BATCH_LATTICES)
        n = _ns(lat)
        out.append(dict(lattice=lat, nup=r.randrange(1, n), ndn=r.randrange(1, n), U=r.uniform(0.0, 12.0)))
    return out


def _batch_starts(case, seed):
    dims = [_dim(q["lattice"], q["nup"], q["ndn"]) for q in _batch_list(case)]
    return list(torch.split(_start(sum(dims), seed), dims))


class _Dense:
    """H of Eq. (1) on a D_up x D_dn matrix: per-spin sparse hopping matrices and the diagonal."""

    def __init__(self, lattice, nup, ndn, U):
        self.T, bits = [], []
        for n in (nup, ndn):
            T, s = self._spin(_ns(lattice), _bonds(lattice), n)
            self.T.append(T)
            bits.append(torch.from_numpy(((s[:, None] >> np.arange(_ns(lattice))) & 1).astype(np.float64)).cuda())
        self.diag = U * (bits[0] @ bits[1].T)
        self.D = self.diag.numel()

    @staticmethod
    def _spin(ns, bonds, n):
        w = np.arange(1 << ns, dtype=np.int64)
        pop = np.zeros_like(w)
        for i in range(ns):
            pop += (w >> i) & 1
        s = w[pop == n]
        rows, cols, vals = [], [], []
        for i, j in bonds:
            k = np.nonzero(((s >> i) ^ (s >> j)) & 1)[0]
            t = s[k] ^ ((1 << i) | (1 << j))
            between = s[k] & (((1 << max(i, j)) - 1) & ~((2 << min(i, j)) - 1))
            rows.append(k)
            cols.append(np.searchsorted(s, t))
            vals.append(np.where(pop[between] & 1, 1.0, -1.0))
        ij = torch.from_numpy(np.stack([np.concatenate(rows), np.concatenate(cols)]))
        T = torch.sparse_coo_tensor(ij, torch.from_numpy(np.concatenate(vals)), (s.size, s.size))
        return T.coalesce().to_sparse_csr().cuda(), s

    def __call__(self, v):
        V = v.reshape(self.diag.shape)
        W = torch.sparse.mm(self.T[1], V.T.contiguous()).T + self.diag * V
        return (W + torch.sparse.mm(self.T[0], V.contiguous())).reshape(-1)


def _krylov(H, v, m, keep=True, done=None):
    """Lanczos from v, every vector orthogonalised against all before it when kept."""
    m = min(m, H.D)
    F = torch.zeros((m if keep else 2, H.D), dtype=torch.float64, device=v.device)
    f, old, a, b = v / v.norm(), torch.zeros_like(v), [], []
    for j in range(m):
        if keep:
            F[j] = f
        w = H(f) - (b[-1] if b else 0.0) * old
        a.append(float(w @ f))
        w -= a[-1] * f
        for _ in range(2 if keep else 0):
            w -= (F[:j + 1] @ w) @ F[:j + 1]
        b.append(float(w.norm()))
        if b[-1] < 1e-11 * max(1.0, max(map(abs, a))) or (done is not None and j % 5 == 4 and done(a, b)):
            break
        f, old = w / b[-1], f
    return np.array(a), np.array(b), F


def _ground(H, v, vector=False):
    def done(a, b):
        T = np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1)
        return b[-1] * abs(np.linalg.eigh(T)[1][-1, 0]) < 1e-13 * max(1.0, abs(a[0]))

    a, b, F = _krylov(H, v, min(400, int(2.4e9 // H.D)), done=done)
    lam, Z = np.linalg.eigh(np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1))
    if not vector:
        return float(lam[0]), None
    s = Z[:, 0] * np.sign(Z[:, 0].sum())          # the sign an iteration started from ones keeps
    return float(lam[0]), torch.from_numpy(np.ascontiguousarray(s)).to(F) @ F[:len(s)]
