"""The work that a user of the library has it do, as cases that can be timed.

A case is a dict of plain values; its "kind" says which entry points it goes through:

  solve      a handle restarted from a start vector (cdfci_set_initial), advanced a number of iterations
             (cdfci_step), its statistics, and the stored vector exported to device arrays and sorted by key
  batch      the same for many uneven problems stepped together (cdfci_batch_step)
  states     xCDFCI: a handle made, advanced, its energies and rows exported, released
  adjoint    dE/dh, dE/dg, dE/dkappa of a loaded vector (cdfci_gradient, RDMs inside)
  quotient   the exact Rayleigh quotient of a loaded vector (cdfci_energy mode 1) and the one under other
             integrals (cdfci_energy_with)
  autograd   CDFCIEnergy forward and backward on integrals that need gradients
  orbitals   OptOrbFCI (cdfci_optorb): outer orbital loop around inner solves

Problems are the repository's own: seeded synthetic ab initio integrals (inputs.synthetic_integrals) and
Hubbard lattices in real space, there with a seeded site and bond disorder, and in momentum space, there with a seeded
start vector.  The electron counts of ab initio problems differ between the spins or the result does not depend
on the choice among mirror images, and the disorder breaks a lattice's symmetry: two coordinates whose
gradients are equal but for the last bit would make a trajectory depend on the order of a sum.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2605_04483_gb300 import api, inputs
from paper_2605_04483_gb300.autograd import CDFCIEnergy

STATS = ("energy", "mu", "alpha", "nnz_c", "n_slots", "elements", "applied", "inserted")


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # The smallest solve: an eight-site chain, one coordinate per step; 32 elements a column, so an
        # iteration is latency alone.
        dict(name="chain8_m1", kind="solve", system="lattice", shape="8", periodic=False, U=4.0, na=4, nb=4, m=1,
             tau=0.0, log2_capacity=16, iterations=1000, rows=4_900),
        # The headline path: Algorithm 1 on the N = 24 integrals of the benchmark, one electron taken out.
        dict(name="ab24_m1", kind="solve", system="ab_initio", N=24, na=6, nb=5, m=1, tau=1e-5, log2_capacity=24,
             iterations=2000, rows=8_000_000),
        # A small molecule-sized space at a block of 64 coordinates, no compression: launches and the
        # reduced problem count here.
        dict(name="ab12_m64", kind="solve", system="ab_initio", N=12, na=4, nb=3, m=64, tau=0.0, log2_capacity=18,
             iterations=48, rows=108_900),
        # Algorithm 2 at the benchmark's block size on the N = 24 integrals: the largest column scatter.
        dict(name="ab24_m128", kind="solve", system="ab_initio", N=24, na=6, nb=5, m=128, tau=1e-4,
             log2_capacity=26, iterations=100, rows=20_000_000),
        # A 4 x 4 lattice in real space at half filling and m = 256: short columns, a large reduced problem.
        dict(name="lattice4x4_m256", kind="solve", system="lattice", shape="4x4", periodic=True, U=8.0, na=8, nb=8,
             m=256, tau=0.0, log2_capacity=24, iterations=200, rows=1_000_000),
        # The same lattice in momentum space, started from the degenerate shell of 400 determinants: 400 forced
        # steps, then Algorithm 1.  (One coordinate a step: every interaction is +-U/L there, so gradients tie, and
        # with a block the ties would fall by the order of the atomic sums.)
        dict(name="momentum4x4_m1", kind="solve", system="lattice_k", shape="4x4", U=4.0, na=8, nb=8, m=1,
             tau=0.0, log2_capacity=22, iterations=1500, rows=1_000_000),
        # Many uneven problems at once, as a scan over molecules and lattices runs them.
        dict(name="batch24", kind="batch", problems=24, mix=4, iterations=32),
        # Four states of the N = 24 problem, from creation to the exported rows.
        dict(name="states4_ab24", kind="states", N=24, na=6, nb=5, states=4, tau=1e-5, log2_capacity=22,
             iterations=400, rows=2_000_000),
        # The energy's derivatives of a large stored vector at the size of the adjoint benchmark.
        dict(name="adjoint16", kind="adjoint", N=16, na=5, nb=5, nonzero=300_000, rows=1_000_000, log2_capacity=21),
        # Exact energies of a stored vector, with odd sizes.
        dict(name="quotient13", kind="quotient", N=13, na=4, nb=3, nonzero=60_000, rows=100_001, log2_capacity=18),
        # A differentiable energy inside a training step: everything from the integrals to their gradients.
        dict(name="autograd9", kind="autograd", N=9, na=4, nb=3, m=1, iterations=400, log2_capacity=16),
        # Orbital optimisation: 9 of 12 orbitals.
        dict(name="orbitals12to9", kind="orbitals", M=12, N=9, na=3, nb=2, outer=2, bb_steps=10, iterations=400,
             log2_capacity=15),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["batch", "states", "adjoint", "adjoint", "quotient", "quotient", "autograd",
                                       "orbitals"])
    if kind == "solve":
        system = rng.choice(["ab_initio", "ab_initio", "lattice", "lattice_k"])
        m = 1 if system == "lattice_k" else rng.choice([1, _log_int(rng, 2, 400)])
        block = lambda dim: max(1, min(m, dim // 16))         # a block is a small part of the space
        if system == "ab_initio":
            N = rng.randint(8, 26)
            na = rng.randint(2, min(6, N - 3))
            nb = max(1, na - rng.randint(1, 2))
            dim = math.comb(N, na) * math.comb(N, nb)
            small = dim < 150_000
            m = block(dim)
            its = rng.randint(200, 1500) if m == 1 else max(8, min(160, 12_000 // m))
            return dict(kind=kind, system=system, N=N, na=na, nb=nb, m=m, tau=0.0 if small else (1e-5 if m == 1 else 1e-4),
                        log2_capacity=18 if small else (24 if m == 1 else 26), iterations=its,
                        rows=min(dim, 8_000_000 if m == 1 else 20_000_000))
        shape = rng.choice(["7", "8", "10", "13", "2x4", "2x5", "3x4", "4x4"] if system == "lattice"
                           else ["2x4", "3x4", "4x4"])
        sites = int(np.prod([int(x) for x in shape.split("x")]))
        na = rng.randint(max(2, sites // 2 - 2), sites // 2)
        nb = na if system == "lattice_k" else rng.randint(max(2, na - 1), na)
        dim = math.comb(sites, na) * math.comb(sites, nb)
        m = block(dim)
        return dict(kind=kind, system=system, shape=shape, periodic=rng.random() < 0.5, U=round(rng.uniform(1.0, 10.0 if system == "lattice" else 4.0), 3),
                    na=na, nb=nb, m=m, tau=0.0, log2_capacity=24, iterations=rng.randint(100, 1000) if m == 1 else
                    rng.randint(20, 120), rows=min(dim, 4_000_000))
    if kind == "batch":
        return dict(kind=kind, problems=rng.randint(2, 24), mix=rng.randint(10, 999), iterations=rng.randint(8, 32))
    if kind == "states":
        N = rng.randint(9, 24)
        na = rng.randint(2, min(6, N - 4))
        return dict(kind=kind, N=N, na=na, nb=na - 1, states=rng.randint(2, 8), tau=1e-5, log2_capacity=22,
                    iterations=_log_int(rng, 20, 400), rows=2_000_000)
    if kind in ("adjoint", "quotient"):
        N = rng.randint(7, 16)
        na = rng.randint(2, 5)
        nb = rng.randint(1, na)
        dim = math.comb(N, na) * math.comb(N, nb)
        nz = min(_log_int(rng, 100, 200_000), max(1, dim // 2))
        rows = min(dim, int(nz * rng.uniform(1.0, 4.0)))
        return dict(kind=kind, N=N, na=na, nb=nb, nonzero=nz, rows=rows,
                    log2_capacity=math.ceil(math.log2((rows + _column_length(N, na, nb)) / 0.7)))
    if kind == "autograd":
        N = rng.randint(6, 12)
        na = rng.randint(2, 4)
        most = math.comb(N, na) * math.comb(N, na - 1) // 16
        return dict(kind=kind, N=N, na=na, nb=na - 1, m=rng.choice([1, max(1, min(rng.randint(4, 64), most))]),
                    iterations=rng.randint(20, 200), log2_capacity=18)
    M = rng.randint(6, 14)
    N = rng.randint(max(5, M - 4), M)
    return dict(kind=kind, M=M, N=N, na=3, nb=2, outer=rng.randint(1, 2), bb_steps=rng.randint(2, 10),
                iterations=rng.randint(50, 400), log2_capacity=16)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _shape(case):
    return tuple(int(x) for x in case["shape"].split("x"))


def _generator(seed):
    return np.random.Generator(np.random.PCG64(int(seed) % (1 << 63)))


def _integrals(case, seed):
    """(h, g, N, reference determinant) of a solve case; reference (0, 0) = chosen by the library."""
    rng = _generator(seed)
    if case["system"] == "ab_initio":
        h, g = inputs.synthetic_integrals(case["N"], rng)
        return h, g, case["N"], (0, 0)
    shape = _shape(case)
    h, g = inputs.hubbard_integrals(shape, 1.0, case["U"], case["periodic"])
    bond = rng.uniform(0.9, 1.1, size=h.shape)
    h = h * 0.5 * (bond + bond.T) + np.diag(rng.uniform(-0.5, 0.0, size=len(h)))
    return h, g, len(h), inputs.neel_reference(shape, case["na"], case["nb"])


def _aufbau(h, na, nb):
    order = sorted(range(len(h)), key=lambda p: (h[p, p], p))
    return sum(1 << p for p in order[:na]), sum(1 << p for p in order[:nb])


def _strings(N, n):
    """Every N-bit word of n ones, ascending."""
    if n == 0:
        return np.zeros(1, dtype=np.int64)
    out, x = [], (1 << n) - 1
    while x < 1 << N:
        out.append(x)
        low = x & -x
        carry = x + low
        x = (((carry ^ x) >> 2) // low) | carry
    return np.array(out, dtype=np.int64)


def _vector(case, h, seed):
    """A CI vector as a selected-CI run leaves it: `rows` determinants of lowest (one-body plus noise) energy,
    the first `nonzero` of them with coefficients that fall off with it.  Returns keys (rows, 2) and c."""
    rng = _generator(seed + 7_919)
    A, B = _strings(case["N"], case["na"]), _strings(case["N"], case["nb"])
    e = np.diag(h)
    bits = lambda X: ((X[:, None] >> np.arange(case["N"])) & 1) @ e
    score = (bits(A)[:, None] + bits(B)[None, :]).ravel()
    score += rng.normal(0.0, 0.5, size=score.size)
    low = np.argpartition(score, case["rows"] - 1)[:case["rows"]]
    low = low[np.argsort(score[low], kind="stable")]
    keys = np.stack([A[low // len(B)], B[low % len(B)]], axis=1).astype(np.uint64)
    c = np.zeros(case["rows"])
    k = np.arange(case["nonzero"])
    c[:case["nonzero"]] = rng.choice([-1.0, 1.0], size=k.size) * rng.uniform(0.5, 1.5, size=k.size) / (1.0 + k) ** 0.6
    return keys, c


def _load(case, h, g, keys, c):
    """A handle that holds the vector: a checkpoint of its rows, restored."""
    s = api.Solver(h, g, case["N"], case["na"], case["nb"], log2_capacity=case["log2_capacity"])
    hdr = api.cdfci_checkpoint_header()
    hdr.version, hdr.N, hdr.n_alpha, hdr.n_beta, hdr.num_coordinates = 1, case["N"], case["na"], case["nb"], 1
    hdr.n_entries = hdr.n_slots = hdr.inserted = len(c)
    hdr.nnz_c = int(np.count_nonzero(c))
    hdr.mu[0], hdr.scale[0] = float(c @ c), 1.0
    s.restore({"header": hdr, "keys": keys, "c": c, "b": np.zeros(len(c)), "flags": None})
    return s


def _batch_cases(case):
    """The problems of a batch: two in three synthetic ab initio (N 12..32, 2..5 electrons a spin, m = 64),
    the others lattices (m = 128)."""
    rng = _generator(104_729 + case["mix"])
    out = []
    for k in range(case["problems"]):
        if k % 3 < 2:
            N, na = int(rng.integers(12, 33)), int(rng.integers(3, 6))
            nb = na - 1
            dim = math.comb(N, na) * math.comb(N, nb)
            out.append(dict(kind="solve", system="ab_initio", N=N, na=na, nb=nb, m=64, tau=0.0 if dim < 500_000 else 1e-3,
                            log2_capacity=20 if dim < 500_000 else 22, rows=min(dim, 1_500_000)))
        else:
            shape = inputs.HUBBARD_SHAPES[int(rng.integers(0, len(inputs.HUBBARD_SHAPES)))]
            N = int(np.prod(shape))
            out.append(dict(kind="solve", system="lattice", shape="x".join(map(str, shape)), periodic=True,
                            U=float(rng.choice([2.0, 4.0, 8.0])), na=N - N // 2, nb=N // 2, m=128, tau=0.0,
                            log2_capacity=20, rows=min(math.comb(N, N // 2) ** 2, 200_000)))
    return out


def _solver(case, seed, stream):
    """The handle of a solve case and its start vector (keys, c)."""
    params = dict(num_coordinates=case["m"], log2_capacity=case["log2_capacity"], z_threshold=case["tau"],
                  cuda_stream=stream.cuda_stream)
    if case["system"] == "lattice_k":
        shape, U = _shape(case), case["U"] * (1.0 + 0.02 * _generator(seed).uniform(-1.0, 1.0))
        s = api.Solver.hubbard_k(shape, case["na"], case["nb"], t=1.0, U=U, **params)
        eps = np.diag(inputs.hubbard_k_integrals(shape, 1.0, U)[0])
        keys = api.cdfci_degenerate_set(eps, case["na"], case["nb"])
        c = 1.0 + _generator(seed + 1).uniform(0.0, 1.0, size=len(keys))
        return s, keys, c / np.linalg.norm(c)
    h, g, N, ref = _integrals(case, seed)
    s = api.Solver(h, g, N, case["na"], case["nb"], ref_alpha=ref[0], ref_beta=ref[1], **params)
    A, B = ref if ref != (0, 0) else _aufbau(h, case["na"], case["nb"])
    return s, np.array([[A, B]], dtype=np.uint64), np.ones(1)


# ---------------------------------------------------------------------------
# Passes
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case, stream=torch.cuda.Stream())
    if kind == "solve":
        s, keys, c = _solver(case, seed, state["stream"])
        state.update(solver=s, keys=keys, c=c)
    elif kind == "batch":
        made = [_solver(p, seed + 31 * k, state["stream"]) for k, p in enumerate(_batch_cases(case))]
        state.update(members=made, batch=api.Batch([s for s, _, _ in made]), problems=_batch_cases(case))
    elif kind == "states":
        h, g = inputs.synthetic_integrals(case["N"], _generator(seed))
        state.update(h=torch.tensor(h, device="cuda"), g=torch.tensor(g, device="cuda"))
    elif kind in ("adjoint", "quotient"):
        rng = _generator(seed)
        h, g = inputs.synthetic_integrals(case["N"], rng)
        state.update(solver=_load(case, h, g, *_vector(case, h, seed)))
        if kind == "quotient":
            h2, g2 = inputs.synthetic_integrals(case["N"], rng)
            state.update(h2=torch.tensor(h2, device="cuda"), g2=torch.tensor(g2, device="cuda"))
    elif kind == "autograd":
        h, g = inputs.synthetic_integrals(case["N"], _generator(seed))
        state.update(h=torch.tensor(h, device="cuda"), g=torch.tensor(g, device="cuda"))
    else:
        h, g = inputs.synthetic_integrals(case["M"], _generator(seed))
        state.update(h=h, g=g)
    torch.cuda.synchronize()
    return state


def _export(s, rows, stream, width=0):
    """The stored vector in device arrays of `rows` rows, ordered by key: codes A | B << N, and c, b (or their
    rows); what is left of the arrays stays zero."""
    n, got = rows, ctypes.c_int64()
    with torch.cuda.stream(stream):
        keys = torch.zeros(n, 2, dtype=torch.int64, device="cuda")
        c = torch.zeros((n, width) if width else n, dtype=torch.float64, device="cuda")
        b = torch.zeros_like(c)
        call = api.lib().cdfci_export_states if width else api.lib().cdfci_export
        api._check(call(s.handle, keys.data_ptr(), c.data_ptr(), b.data_ptr(), n, ctypes.byref(got)))
        codes, order = torch.sort(keys[:, 0] | (keys[:, 1] << s.N))
        return dict(codes=codes, c=c[order], b=b[order])


def _pick(st):
    return {k: np.float64(st[k]) if isinstance(st[k], float) else st[k] for k in STATS}


def run(state):
    case, stream = state["case"], state["stream"]
    kind = case["kind"]
    if kind == "solve":
        s = state["solver"]
        s.set_initial(state["keys"], state["c"])
        st = s.step(case["iterations"])
        return dict(stats=_pick(st), vector=_export(s, case["rows"], stream))
    if kind == "batch":
        for s, keys, c in state["members"]:
            s.set_initial(keys, c)
        sts = state["batch"].step(case["iterations"])
        every = [_export(s, p["rows"], stream) for (s, _, _), p in zip(state["members"], state["problems"])]
        with torch.cuda.stream(stream):
            return dict(stats={k: np.array([st[k] for st in sts]) for k in STATS},
                        vectors={k: torch.cat([v[k] for v in every]) for k in ("codes", "c", "b")})
    if kind == "states":
        s = api.Solver(state["h"], state["g"], case["N"], case["na"], case["nb"], num_states=case["states"],
                       z_threshold=case["tau"], log2_capacity=case["log2_capacity"], cuda_stream=stream.cuda_stream)
        try:
            st = s.step(case["iterations"])
            return dict(energies=s.energies(), elements=st["elements"], applied=st["applied"],
                        rows=_export(s, case["rows"], stream, case["states"]))
        finally:
            s.close()
    if kind == "adjoint":
        dh, dg, dk = state["solver"].gradient()
        return dict(dh=dh, dg=dg, dkappa=dk)
    if kind == "quotient":
        s = state["solver"]
        return dict(E=np.float64(s.energy(1)), E_with=np.float64(s.energy_with(state["h2"], state["g2"])))
    if kind == "autograd":
        h, g = state["h"].detach().requires_grad_(), state["g"].detach().requires_grad_()
        E = CDFCIEnergy.apply(h, g, case["N"], case["na"], case["nb"], case["iterations"],
                              dict(num_coordinates=case["m"], log2_capacity=case["log2_capacity"]))
        E.backward()
        return dict(E=E.detach(), dh=h.grad, dg=g.grad)
    U, E = api.cdfci_optorb(state["h"], state["g"], case["M"], case["N"], case["na"], case["nb"], outer=case["outer"],
                            bb_steps=case["bb_steps"], inner_iterations=case["iterations"],
                            log2_capacity=case["log2_capacity"])
    return dict(U=U, E=E)


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _column_length(N, na, nb):
    va, vb = N - na, N - nb
    return (1 + na * va + nb * vb + math.comb(na, 2) * math.comb(va, 2) + math.comb(nb, 2) * math.comb(vb, 2)
            + na * va * nb * vb)


def _elements(case):
    """Matrix elements of one column that can be nonzero."""
    if case["system"] == "ab_initio":
        return _column_length(case["N"], case["na"], case["nb"])
    N = int(np.prod(_shape(case)))
    if case["system"] == "lattice":
        return 1 + 2 * (case["na"] + case["nb"])
    return 1 + case["na"] * case["nb"] * (N - max(case["na"], case["nb"]))


def _solve_work(case, iterations):
    """Each element reads its key, c and b and writes b (40 bytes); a value is an integral times the step."""
    n = _elements(case) * case["m"] * iterations
    cube = 0 if case["m"] == 1 else 20 * (case["m"] + 1) ** 2 * iterations
    return 40 * n, 4 * n + cube


def work(case):
    kind = case["kind"]
    if kind == "solve":
        b, f = _solve_work(case, case["iterations"])
    elif kind == "batch":
        parts = [_solve_work(p, case["iterations"]) for p in _batch_cases(case)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "states":
        n = _column_length(case["N"], case["na"], case["nb"]) * case["iterations"]
        b, f = (16 + 24 * case["states"]) * n, 4 * case["states"] * n
    elif kind == "adjoint":
        b = 32 * case["rows"] + 8 * 3 * case["N"] ** 4
        f = 2 * case["nonzero"] * _column_length(case["N"], case["na"], case["nb"])
    elif kind == "quotient":
        b = 2 * (32 * case["rows"] + 8 * case["N"] ** 4)
        f = 2 * 2 * case["nonzero"] * _column_length(case["N"], case["na"], case["nb"])
    elif kind == "autograd":
        n = _column_length(case["N"], case["na"], case["nb"]) * case["m"] * case["iterations"]
        b, f = 40 * n + 8 * 3 * case["N"] ** 4, 4 * n
    else:
        n = _column_length(case["N"], case["na"], case["nb"]) * case["iterations"] * case["outer"]
        M, N = case["M"], case["N"]
        turns = case["outer"] * (case["bb_steps"] + 1)
        b = 40 * n + turns * 8 * M ** 4
        f = 4 * n + turns * 2 * (M ** 4 * N + M ** 3 * N ** 2 + M ** 2 * N ** 3 + M * N ** 4)
    return {"bytes": int(b), "flops": int(f)}


# ---------------------------------------------------------------------------
# The same results in plain numpy, 64 bits
# ---------------------------------------------------------------------------

class _Plain:
    """Algorithms 1 and 2 from the reference determinant, written out over numpy columns."""

    def __init__(self, h, g, na, nb, tau):
        self.h, self.g, self.N, self.tau = h, g, len(h), tau
        self.index, self.code = {}, []
        self.c, self.b = np.zeros(0), np.zeros(0)
        self.J = np.einsum("ppqq->pq", g)
        self.K = np.einsum("pqqp->pq", g)
        self.cache = {}

    def diagonal(self, A, B):
        a, b = self._occ(A), self._occ(B)
        e = self.h[a, a].sum() + self.h[b, b].sum()
        for x in (a, b):
            e += 0.5 * (self.J[np.ix_(x, x)] - self.K[np.ix_(x, x)]).sum()
        return e + self.J[np.ix_(a, b)].sum()

    def _occ(self, X):
        return np.array([p for p in range(self.N) if X >> p & 1], dtype=np.int64)

    def _string(self, X):
        """Singles and same-spin doubles of one string: orbitals, signs and changed strings."""
        N, occ = self.N, self._occ(X)
        vir = np.array([p for p in range(N) if not X >> p & 1], dtype=np.int64)
        below = np.cumsum([0] + [X >> p & 1 for p in range(N)])[:N]
        cross = lambda i, a: np.where(a > i, below[a] - below[i] - 1, below[i] - below[a])
        bit = np.uint64(1) << np.arange(N, dtype=np.uint64)
        i, a = (x.ravel() for x in np.meshgrid(occ, vir, indexing="ij"))
        singles = (i, a, 1.0 - 2.0 * (cross(i, a) & 1), np.uint64(X) ^ bit[i] ^ bit[a])
        oi, oj = np.triu_indices(len(occ), 1)
        va, vb = np.triu_indices(len(vir), 1)
        i, a = (x.ravel() for x in np.meshgrid(occ[oi], vir[va], indexing="ij"))
        j, b = (x.ravel() for x in np.meshgrid(occ[oj], vir[vb], indexing="ij"))
        between = lambda p, x, y: ((p > np.minimum(x, y)) & (p < np.maximum(x, y))).astype(np.int64)
        moved = cross(i, a) + cross(j, b) - between(i, j, b) + between(a, j, b)
        doubles = (i, a, j, b, 1.0 - 2.0 * (moved & 1), np.uint64(X) ^ bit[i] ^ bit[a] ^ bit[j] ^ bit[b])
        return occ, singles, doubles

    def column(self, code):
        """Codes and values of the off-diagonal elements that are not zero."""
        if code in self.cache:
            return self.cache[code]
        N, h, g = self.N, self.h, self.g
        A, B = code & ((1 << N) - 1), code >> N
        (oa, sa, da), (ob, sb, db) = self._string(A), self._string(B)
        codes, vals = [], []
        put = lambda x, y: x | (y << np.uint64(N))
        for alpha, (i, a, sg, X) in ((True, sa), (False, sb)):
            same, other = (oa, ob) if alpha else (ob, oa)
            v = h[i, a] + (g[i[:, None], a[:, None], same, same] - g[i[:, None], same, same, a[:, None]]).sum(1)
            v = v + g[i[:, None], a[:, None], other, other].sum(1)
            codes.append(put(X, np.uint64(B)) if alpha else put(np.uint64(A), X))
            vals.append(sg * v)
        for alpha, (i, a, j, b, sg, X) in ((True, da), (False, db)):
            codes.append(put(X, np.uint64(B)) if alpha else put(np.uint64(A), X))
            vals.append(sg * (g[i, a, j, b] - g[i, b, j, a]))
        codes.append(put(sa[3][:, None], sb[3][None, :]).ravel())
        vals.append((sa[2][:, None] * sb[2] * g[sa[0][:, None], sa[1][:, None], sb[0], sb[1]]).ravel())
        codes, vals = np.concatenate(codes), np.concatenate(vals)
        keep = vals != 0.0
        got = self.cache[code] = (codes[keep].tolist(), vals[keep])
        return got

    def entry(self, code):
        k = self.index.get(code)
        if k is None:
            k = self.index[code] = len(self.code)
            self.code.append(code)
            if k >= len(self.c):
                self.c, self.b = np.resize(self.c, 2 * k + 1024), np.resize(self.b, 2 * k + 1024)
            self.c[k] = self.b[k] = 0.0
        return k

    def scatter(self, code, eta):
        """b += eta H_{:,code} with the compression rule; the rows updated, sum_j H_ji c_j."""
        codes, H = self.column(code)
        v = eta * H
        at = np.array([self.index.get(x, -1) for x in codes], dtype=np.int64)
        for k in np.flatnonzero((at < 0) & (np.abs(v) >= self.tau)):
            at[k] = self.entry(codes[k])
        c = np.where(at >= 0, self.c[at], 0.0)
        on = (at >= 0) & ((c != 0.0) | (np.abs(v) >= self.tau))
        self.b[at[on]] += v[on]
        return at[on], float(H @ c)

    def start(self, code):
        k = self.entry(code)
        self.c[k] = 1.0
        rows, _ = self.scatter(code, 1.0)
        A, B = code & ((1 << self.N) - 1), code >> self.N
        self.b[k] = self.diagonal(A, B)
        self.mu, self.alpha = 1.0, float(self.b[k])
        self.candidates = np.append(rows, k)

    def _ordered(self):
        """The candidates, the smaller key first (among equal gradients it is chosen)."""
        cand = np.unique(self.candidates)
        return cand[np.argsort(np.array([self.code[k] for k in cand], dtype=np.uint64), kind="stable")]

    def _diag(self, k):
        return self.diagonal(self.code[k] & ((1 << self.N) - 1), self.code[k] >> self.N)

    def step1(self):
        cand = self._ordered()
        k = int(cand[np.argmax(np.abs(self.b[cand] + self.mu * self.c[cand]))])
        ci, bi, Hii = self.c[k], self.b[k], self._diag(k)
        v1, v2, v3 = 4.0 * bi + 4.0 * self.mu * ci, 2.0 * Hii + 4.0 * ci * ci + 2.0 * self.mu, 4.0 * ci
        roots = np.roots([4.0, 3.0 * v3, 2.0 * v2, v1])
        roots = np.sort(roots[np.abs(roots.imag) <= 1e-7 * (1.0 + np.abs(roots))].real)
        for _ in range(4):                                    # Newton steps on the cubic
            f = ((4.0 * roots + 3.0 * v3) * roots + 2.0 * v2) * roots + v1
            d = (12.0 * roots + 6.0 * v3) * roots + 2.0 * v2
            roots = roots - np.where(d != 0.0, f / np.where(d != 0.0, d, 1.0), 0.0)
        eta = roots[0]
        if len(roots) == 3 and (roots[2] - roots[1]) - (roots[1] - roots[0]) > 1e-9 * (roots[2] - roots[0]):
            eta = roots[2]
        self.c[k] = ci + eta
        rows, gathered = self.scatter(self.code[k], eta)
        self.mu += 2.0 * eta * ci + eta * eta
        self.alpha += 2.0 * eta * bi + eta * eta * Hii
        self.b[k] = Hii * self.c[k] + gathered
        self.candidates = np.append(rows, k)

    def step(self, m):
        cand = self._ordered()
        grad = np.abs(self.b[cand] + self.mu * self.c[cand])
        I = cand[np.argsort(-grad, kind="stable")[:m]]
        codes = [self.code[k] for k in I]
        where = {x: t for t, x in enumerate(codes)}
        H = np.diag([self._diag(k) for k in I])
        for t, x in enumerate(codes):
            col, vals = self.column(x)
            for y, v in zip(col, vals):
                s = where.get(y)
                if s is not None:
                    H[s, t] = v
        cI, bI = self.c[I].copy(), self.b[I].copy()
        lone = np.count_nonzero(self.c[:len(self.code)]) == np.count_nonzero(cI)
        if lone:
            lam, V = np.linalg.eigh(H)
            z, gamma = V[:, 0] * math.sqrt(-lam[0]), 1.0
            if z @ cI < 0.0:
                z = -z
        else:
            nu = math.sqrt(self.mu - cI @ cI)
            R = np.zeros((len(I) + 1, len(I) + 1))
            R[0, 0] = (self.alpha - 2.0 * cI @ bI + cI @ H @ cI) / nu ** 2
            R[0, 1:] = R[1:, 0] = (bI - H @ cI) / nu
            R[1:, 1:] = H
            lam, V = np.linalg.eigh(R)
            z = V[:, 0] * math.sqrt(-lam[0])
            if z[0] < 0.0:
                z = -z
            gamma, z = z[0] / nu, z[1:]
        eta = z - gamma * cI
        n = len(self.code)
        self.c[:n] *= gamma
        self.b[:n] *= gamma
        self.c[I] = z
        done = [self.scatter(x, e) for x, e in zip(codes, eta)]
        self.mu = gamma ** 2 * self.mu + 2.0 * gamma * eta @ cI + eta @ eta
        self.alpha = gamma ** 2 * self.alpha + 2.0 * gamma * eta @ bI + eta @ H @ eta
        for t, k in enumerate(I):                             # the gather after every insertion changes nothing:
            self.b[k] = H[t, t] * self.c[k] + done[t][1]      # a new row has c = 0
        self.candidates = np.concatenate([rows for rows, _ in done] + [I])

    def solve(self, code, m, iterations):
        self.start(code)
        for _ in range(iterations):
            if m == 1:
                self.step1()
            else:
                self.step(m)
        n = len(self.code)
        codes = np.array(self.code, dtype=np.uint64)
        order = np.argsort(codes, kind="stable")
        return codes[order], self.c[:n][order], self.b[:n][order]


def _density(N, na, nb, codes, c):
    """Spin-summed gamma and Gamma of a vector over determinants A | B << N, from E_rs |c> in the full space."""
    A, B = _strings(N, na), _strings(N, nb)
    C = np.zeros((len(A), len(B)))
    codes = codes.astype(np.uint64)
    low = np.uint64((1 << N) - 1)
    C[np.searchsorted(A, (codes & low).astype(np.int64)), np.searchsorted(B, (codes >> np.uint64(N)).astype(np.int64))] = c
    V = np.zeros((N, N) + C.shape)
    for X, axis in ((A, 0), (B, 1)):
        for p in range(N):
            for q in range(N):
                at = np.flatnonzero((X >> q & 1) & ((X >> p & 1) ^ 1)) if p != q else np.flatnonzero(X >> p & 1)
                if not len(at):
                    continue
                lo, hi = min(p, q), max(p, q)
                mask = (1 << hi) - (1 << (lo + 1)) if hi > lo else 0
                sign = np.array([1.0 - 2.0 * (bin(int(x) & mask).count("1") & 1) for x in X[at]])
                to = np.searchsorted(X, X[at] ^ (1 << p) ^ (1 << q)) if p != q else at
                if axis == 0:
                    V[p, q][to] += sign[:, None] * C[at]
                else:
                    V[p, q][:, to] += sign * C[:, at]
    V = V.reshape(N * N, -1)
    g1 = (V @ C.ravel()).reshape(N, N)
    G = (V @ V.T).reshape(N, N, N, N).transpose(1, 0, 2, 3).copy()     # <c|E_pq E_rs|c> = <E_qp c|E_rs c>
    for q in range(N):
        G[:, q, q, :] -= g1
    norm = C.ravel() @ C.ravel()
    return 0.5 * (g1 + g1.T) / norm, G / norm


def _gradients(h, g, g1, G2):
    s = G2 + G2.transpose(1, 0, 2, 3)
    s = s + s.transpose(0, 1, 3, 2)
    dg = 0.0625 * (s + s.transpose(2, 3, 0, 1))
    F = h @ g1.T + np.einsum("prst,qrst->pq", g, G2, optimize=True)
    return g1, dg, 2.0 * (F - F.T)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        if case["system"] == "lattice_k":
            return None
        N = case["N"] if case["system"] == "ab_initio" else int(np.prod(_shape(case)))
        n = _column_length(N, case["na"], case["nb"])
        if case["iterations"] * case["m"] * n > 6_000_000 or 2 * N > 62:
            return None
        h, g, N, ref = _integrals(case, seed)
        A, B = ref if ref != (0, 0) else _aufbau(h, case["na"], case["nb"])
        p = _Plain(h, g, case["na"], case["nb"], case["tau"])
        _, c, b = p.solve(A | B << N, case["m"], case["iterations"])
        stats = dict(energy=np.float64(p.alpha / p.mu), mu=np.float64(p.mu), alpha=np.float64(p.alpha))
        fill = np.zeros(case["rows"] - len(c))                # unused rows (code 0) sort first
        return dict(stats={k: stats.get(k) for k in STATS},
                    vector=dict(codes=None, c=np.concatenate([fill, c]), b=np.concatenate([fill, b])))
    if kind == "autograd":
        if case["iterations"] * case["m"] * _column_length(case["N"], case["na"], case["nb"]) > 3_000_000:
            return None
        h, g = inputs.synthetic_integrals(case["N"], _generator(seed))
        A, B = _aufbau(h, case["na"], case["nb"])
        codes, c, _ = _Plain(h, g, case["na"], case["nb"], 0.0).solve(A | B << case["N"], case["m"], case["iterations"])
        g1, G2 = _density(case["N"], case["na"], case["nb"], codes, c)
        dh, dg, _ = _gradients(h, g, g1, G2)
        return dict(E=np.float64((h * g1).sum() + 0.5 * (g * G2).sum()), dh=dh, dg=dg)
    if kind in ("adjoint", "quotient"):
        N = case["N"]
        if N * N * math.comb(N, case["na"]) * math.comb(N, case["nb"]) > 120_000_000:
            return None
        rng = _generator(seed)
        h, g = inputs.synthetic_integrals(N, rng)
        keys, c = _vector(case, h, seed)
        g1, G2 = _density(N, case["na"], case["nb"], keys[:, 0] | (keys[:, 1] << np.uint64(N)), c)
        if kind == "adjoint":
            return dict(zip(("dh", "dg", "dkappa"), _gradients(h, g, g1, G2)))
        energy = lambda h, g: np.float64((h * g1).sum() + 0.5 * (g * G2).sum())
        return dict(E=energy(h, g), E_with=energy(*inputs.synthetic_integrals(N, rng)))
    return None
