"""The work that users of this library have it do, as cases that can be timed and checked.

A case is one call sequence through the public entry points (``librpa_gpu``): whole RPA energies
(response function + correlation energy) in the precision modes that are in use, the response function alone with
its matrices, the correlation energy alone, a batch of structures and the no-allocation energy
integrand.  Structures: the two-atom cubic cell, random cells of three species (5/9/13 NAO, 20/40/60
auxiliary functions per atom) at the density of the cubic cell, and the graphene 4x4 slab with a
water-shaped molecule (35 atoms, N_aux 2010); k-meshes from one point to 4x4x1, 6 to 16 tau points.

``listed`` names the cases, ``draw`` gives more of the same ranges, ``prepare`` builds what a program
holds before the call (filled handles), ``run`` makes one pass, ``work`` counts what a pass cannot do
without, ``exact`` evaluates the same quantities in 64 bits as a sum over Kohn-Sham states.
"""
import functools
import itertools
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_2407_19930_gb300 import librpa_gpu as L

MODES = {"fp64": L.LIBRPA_FP64, "fp64_tc": L.LIBRPA_FP64_TC, "split": L.LIBRPA_SPLIT}
R_CUT = 6.0                                        # LRI cutoff (bohr)
SPECIES = [(5, 20, 1), (9, 40, 2), (13, 60, 2)]    # (NAO, auxiliary functions, occupied bands) per atom


def _case(name, call, cell, mode, kmesh=(1, 1, 1), ntau=8, natoms=2, geom=0, spins=1, screen=0.0):
    c = {"call": call, "cell": cell, "mode": mode, "k1": kmesh[0], "k2": kmesh[1], "k3": kmesh[2], "ntau": ntau,
         "natoms": natoms, "geom": geom, "spins": spins, "screen": screen}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest request: a two-atom cell on a 2x2x2 mesh, as in a convergence test or a scan over many
        # cells; the default FP64 mode and the FP64-accurate tensor-core mode
        _case("cubic_fp64", "energy", "cubic", "fp64", (2, 2, 2), 8),
        _case("cubic_tc", "energy", "cubic", "fp64_tc", (2, 2, 2), 8),
        # a spin-polarised cell of a few atoms of several species (ragged blocks, two channels)
        _case("spin_fp64", "energy", "random", "fp64", (2, 2, 1), 8, natoms=4, geom=1, spins=2),
        # a middle-sized cell, as a served request
        _case("cell_tc", "energy", "random", "fp64_tc", (2, 2, 1), 16, natoms=21, geom=2),
        # the response function alone, its matrices taken by a program on the GPU; odd mesh, 12 points
        _case("chi0_tc", "chi0", "random", "fp64_tc", (3, 3, 1), 12, natoms=9, geom=3),
        # the correlation energy alone, repeated with new Coulomb matrices on a finished response function
        _case("ec_fp64", "ec", "random", "fp64", (3, 2, 1), 12, natoms=12, geom=4),
        # a slab of 35 atoms with one k point: a molecule-like calculation in the default mode
        _case("slab_fp64", "energy", "slab", "fp64", (1, 1, 1), 8),
        # the adsorption workload: graphene slab and molecule, 4x4x1 mesh, 16 points (the largest request)
        _case("slab_tc", "energy", "slab", "fp64_tc", (4, 4, 1), 16),
        # the same slab on a coarser mesh in the mixed mode
        _case("slab_split", "energy", "slab", "split", (2, 2, 1), 16),
        # production screening of the Green's functions (threshold 1e-3), odd mesh
        _case("slab_screened", "energy", "slab", "fp64_tc", (3, 3, 1), 12, screen=1e-3),
        # many small structures in one pass, mixed mode (a data set of cells)
        _case("batch_split", "batch", "random", "split", (2, 2, 1), 8, natoms=6, geom=5),
        # host codes that own all device memory: the integrand of one q point without any allocation
        _case("noalloc", "noalloc", "matrix", "fp64", natoms=180, ntau=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo - 0.49), math.log(hi + 0.49)))))


def draw(rng):
    """One more case: sizes over the whole range (log-uniform), cost bounded by the largest listed one."""
    kind = rng.choice(["energy", "energy", "energy", "energy", "slab", "chi0", "ec", "batch", "noalloc"])
    geom = rng.randrange(1000)
    if kind == "noalloc":
        return _case("", "noalloc", "matrix", "fp64", natoms=_log(rng, 16, 300), ntau=rng.randrange(4, 17))
    ntau = rng.choice([6, 8, 10, 12, 14, 16])
    mode = rng.choice(["fp64", "fp64_tc", "fp64_tc", "split"])
    spins = 2 if kind == "energy" and rng.random() < 0.25 else 1
    screen = 1e-3 if kind in ("energy", "slab") and rng.random() < 0.15 else 0.0
    meshes = [(1, 1, 1), (2, 1, 1), (2, 2, 1), (3, 2, 1), (3, 3, 1), (2, 2, 2), (4, 3, 1), (4, 4, 1)]
    kmesh = rng.choice(meshes)
    if kind == "slab":
        kmesh = (1, 1, 1) if mode == "fp64" else rng.choice([m for m in meshes if m[2] == 1])
        if mode == "fp64":
            ntau = min(ntau, 10)
        return _case("", "energy", "slab", mode, kmesh, ntau, screen=screen)
    if rng.random() < 0.15 and kind == "energy":
        return _case("", "energy", "cubic", mode, rng.choice([(2, 2, 2), (3, 1, 2), (2, 2, 1)]), ntau, spins=spins)
    natoms = _log(rng, 2, 32)
    if kind == "batch":
        natoms = min(natoms, 8)
        kmesh = rng.choice(meshes[:4])
    limit = {"energy": 1.0e12, "chi0": 1.0e12, "ec": 0.5e12, "batch": 0.8e12}[kind] * (1.0 if mode == "fp64" else 3.0)
    while True:   # fewer atoms until the pass fits
        c = _case("", kind, "random", mode, kmesh, ntau, natoms=natoms, geom=geom, spins=spins, screen=screen)
        nbytes = np.prod(kmesh) * ntau * 16.0 * (40.0 * natoms) ** 2
        # the correlation energy alone needs a response function first: its cost counts as well
        if natoms <= 2 or (work(dict(c, call="energy") if kind == "ec" else c)["flops"] < limit and
                           (kind != "chi0" or nbytes < 4e9)):
            return c
        natoms -= 1 + natoms // 8


# ------------------------------------------------------------------ structures and inputs


class _Structure:
    def __init__(self, lat, pos, species, kmesh, spins):
        self.lat, self.pos, self.kmesh, self.nspins = np.asarray(lat, float), np.asarray(pos, float), kmesh, spins
        self.n_ao, self.n_aux, self.n_low = (np.array([s[x] for s in species]) for x in range(3))
        self.nat, self.nao, self.naux = len(species), int(self.n_ao.sum()), int(self.n_aux.sum())
        self.nk, self.nocc = int(np.prod(kmesh)), int(self.n_low.sum())
        self.off = np.concatenate([[0], np.cumsum(self.n_ao)])
        self.xoff = np.concatenate([[0], np.cumsum(self.n_aux)])

    def pairs_within(self, rmax):
        """(I, J, R, distance) of every J in cell R within rmax of I in the home cell."""
        inv = np.linalg.inv(self.lat)
        b = [int(math.ceil(rmax * np.linalg.norm(inv[:, a]))) + 1 for a in range(3)]
        R = np.array(list(itertools.product(*[range(-x, x + 1) for x in b])))
        d = np.linalg.norm(self.pos[None, :, None] + (R @ self.lat)[None, None] - self.pos[:, None, None], axis=-1)
        I, J, r = np.nonzero(d <= rmax)
        return I, J, R[r], d[I, J, r]


def _slab(kmesh, spins):
    a = 4.65
    a1, a2 = np.array([a, 0.0, 0.0]), np.array([a / 2, a * math.sqrt(3) / 2, 0.0])
    z0 = np.array([0.0, 0.0, 10.0])
    pos = [i * a1 + j * a2 + s * (a1 + a2) / 3.0 + z0 for i in range(4) for j in range(4) for s in (0, 1)]
    o = (a1 + a2) * 2.0 / 3.0 + z0 + np.array([0.0, 0.0, 6.0])
    t = math.radians(104.5) / 2
    pos += [o, o + 1.81 * np.array([math.sin(t), 0.0, -math.cos(t)]), o + 1.81 * np.array([-math.sin(t), 0.0, -math.cos(t)])]
    species = [(13, 60, 2)] * 32 + [(5, 30, 2), (5, 30, 1), (5, 30, 1)]
    return _Structure([4 * a1, 4 * a2, [0.0, 0.0, 30.0]], pos, species, kmesh, spins)


def _random_cell(natoms, geom, kmesh, spins):
    rng = np.random.default_rng([77, natoms, geom])
    l = (natoms * 32.0) ** (1.0 / 3.0)
    lat = np.eye(3) * l + rng.uniform(-0.1, 0.1, (3, 3)) * l * np.array([[0, 1, 1], [0, 0, 1], [0, 0, 0]])
    cells = np.array(list(itertools.product((-1, 0, 1), repeat=3))) @ lat
    pos, gap = [], 2.5
    while len(pos) < natoms:
        p = rng.uniform(0, 1, 3) @ lat
        if all(np.linalg.norm(p - q + cells, axis=1).min() >= gap for q in pos):
            pos.append(p)
        gap *= 0.9998   # always ends
    return _Structure(lat, pos, [SPECIES[int(x)] for x in rng.integers(0, 3, natoms)], kmesh, spins)


@functools.lru_cache(maxsize=64)
def _structure_of(cell, natoms, geom, kmesh, spins):
    if cell == "slab":
        return _slab(kmesh, spins)
    if cell == "cubic":
        return _Structure(np.eye(3) * 4.0, [[0.0] * 3, [2.0] * 3], [(8, 24, 2)] * 2, kmesh, spins)
    return _random_cell(natoms, geom, kmesh, spins)


def _structures(case):
    """The structure of the case, or those of its batch: eight cells around the stated size."""
    kmesh = (case["k1"], case["k2"], case["k3"])
    n, g = case["natoms"], case["geom"]
    if case["call"] != "batch":
        return [_structure_of(case["cell"], n, g, kmesh, case["spins"])]
    sizes = [max(1, n + d) for d in (-3, -2, -1, 0, 0, 1, 2, 3)]
    return [_structure_of("random", m, 10 * g + i, kmesh, 1) for i, m in enumerate(sizes)]


def _kfrac(kmesh):
    return np.array(list(itertools.product(*[range(n) for n in kmesh])), float) / np.array(kmesh)


def _minus(kmesh):
    n1, n2, n3 = kmesh
    return [(((-a) % n1) * n2 + (-b) % n2) * n3 + (-c) % n3
            for a, b, c in itertools.product(range(n1), range(n2), range(n3))]


def _kohn_sham(st, rng, t0):
    """Tight-binding Kohn-Sham data per spin channel: [(eig, occ, wfc)] and the gap's edges.  On-site levels at
    -0.5 / +0.5 Ha, hoppings that decay with the distance; real H(R), so that c(-k) = conj c(k)."""
    I, J, R, d = st.pairs_within(9.0)
    keep = [x for x in range(len(I)) if I[x] < J[x] or (I[x] == J[x] and tuple(R[x]) > (0, 0, 0))]
    hop = {}
    for x in keep:
        i, j = int(I[x]), int(J[x])
        t = t0 * rng.standard_normal((st.n_ao[i], st.n_ao[j])) * math.exp(-d[x] / 1.5)
        for key, r, c, v in ((tuple(R[x]), i, j, t), (tuple(-R[x]), j, i, t.T)):
            h = hop.setdefault(key, np.zeros((st.nao, st.nao)))
            h[st.off[r]:st.off[r + 1], st.off[c]:st.off[c + 1]] += v
    base = np.concatenate([np.where(np.arange(n) < l, -0.5, 0.5) for n, l in zip(st.n_ao, st.n_low)])
    kf, mi = _kfrac(st.kmesh), _minus(st.kmesh)
    out = []
    for s in range(st.nspins):
        site, nocc = base.copy(), st.nocc
        if st.nspins == 2 and s == 0:   # one more occupied orbital on atom 0 in the first channel
            site[st.n_low[0]] = -0.5
            nocc += 1

        def solve(ik):
            h = np.diag(site).astype(complex)
            for r, b in hop.items():
                h += np.exp(2j * np.pi * float(kf[ik] @ np.array(r))) * b
            h = 0.5 * (h + h.conj().T)
            w, v = np.linalg.eigh(h.real if mi[ik] == ik else h)
            return w, np.ascontiguousarray(v.T.astype(complex))

        todo = [k for k in range(st.nk) if k <= mi[k]]
        with ThreadPoolExecutor(8) as ex:
            done = dict(zip(todo, ex.map(solve, todo)))
        eig = np.array([done[min(k, mi[k])][0] for k in range(st.nk)])
        wfc = np.array([done[k][1] if k in done else done[mi[k]][1].conj() for k in range(st.nk)])
        occ = np.zeros_like(eig)
        occ[:, :nocc] = 1.0
        out.append((eig, occ, wfc))
    edge = [(e[o > 0].max(), e[o < 1].min()) for e, o, _ in out]
    return out, max(x[0] for x in edge), min(x[1] for x in edge)


def _coulomb(st, gen, scale, device):
    """V(q) = scale (A A^H + 0.1 I) on the device, V(-q) = conj V(q), real at q = -q."""
    mi, n = _minus(st.kmesh), st.naux
    v = torch.empty((st.nk, n, n), dtype=torch.complex128, device=device)
    for q in range(st.nk):
        p = mi[q]
        if p < q:
            v[q] = v[p].conj()
        elif p == q:
            a = torch.randn((n, n), dtype=torch.float64, device=device, generator=gen) / math.sqrt(n)
            v[q] = scale * (a @ a.T + 0.1 * torch.eye(n, dtype=torch.float64, device=device))
        else:
            a = torch.randn((n, n), dtype=torch.complex128, device=device, generator=gen) / math.sqrt(n)
            w = a @ a.conj().T
            v[q] = scale * (0.5 * (w + w.conj().T) + 0.1 * torch.eye(n, dtype=torch.float64, device=device))
    return v


def _grid(n, dmin, dmax):
    """Gauss-Legendre points mapped to (0, inf), and the matrix of the cosine transform fitted over the
    transition energies."""
    t, w = np.polynomial.legendre.leggauss(n)
    w0 = math.sqrt(dmin * dmax)
    omega = w0 * (1 + t) / (1 - t)
    tau = (1 + t) / (1 - t) / w0
    e = np.geomspace(dmin, dmax, 400)
    basis = np.exp(-np.outer(e, tau))
    gamma = np.empty((n, n))
    for k in range(n):
        f = 2 * e / (e * e + omega[k] ** 2)
        gamma[k] = np.linalg.lstsq(basis / f[:, None], np.ones(len(e)), rcond=1e-9)[0]
    return dict(tau=tau, omega=omega, w_omega=2 * w0 * w / (1 - t) ** 2, gamma=gamma)


class _Inputs:
    """Everything one request passes in, from the structure and the seed."""

    def __init__(self, st, case, seed, index=0):
        rng = np.random.default_rng([seed, index, 20240719])
        device = "cuda" if torch.cuda.is_available() else "cpu"
        gen = torch.Generator(device=device)
        gen.manual_seed(int(rng.integers(1 << 40)))
        self.st, t0 = st, 0.1
        for _ in range(30):
            self.ks, top, bottom = _kohn_sham(st, rng, t0)
            if bottom - top >= 0.1:
                break
            t0 *= 0.8
        self.efermi = 0.5 * (top + bottom)
        self.lri = []
        for I, K, R, d in zip(*st.pairs_within(R_CUT)):
            c = rng.standard_normal((st.n_aux[I], st.n_ao[I], st.n_ao[K])) * math.exp(-d / 2.0)
            if I == K and not R.any():
                c = 0.5 * (c + c.transpose(0, 2, 1))
            self.lri.append((int(I), int(K), tuple(int(x) for x in R), np.ascontiguousarray(c)))
        self.v = _coulomb(st, gen, {"slab": 3e-4, "cubic": 1e-3}.get(case["cell"], 2e-4), device)
        # the slab takes the library's own grid (it is built from the spectrum), the others bring theirs
        self.grid = None
        if case["cell"] != "slab" or st.nk == 1:
            lo = min(e[o < 1].min() - e[o > 0].max() for e, o, _ in self.ks)
            hi = max(e[o < 1].max() - e[o > 0].min() for e, o, _ in self.ks)
            self.grid = _grid(case["ntau"], lo, hi)


# ------------------------------------------------------------------ states


class _State:
    def __init__(self, case):
        self.case, self.handles, self.batch, self.keep = case, [], None, []

    def __del__(self):
        try:
            L.librpa_gpu_batch_destroy(self.batch)
            for h in self.handles:
                L.librpa_gpu_destroy(h)
        except Exception:   # at interpreter exit
            pass


def _handle(case, inp, stream):
    st = inp.st
    o = L.librpa_gpu_default_opts()
    o.precision, o.n_tau = MODES[case["mode"]], case["ntau"]
    h = L.librpa_gpu_create(o, torch_stream=stream)
    L.librpa_gpu_set_structure(h, st.lat, st.pos, st.n_ao, st.n_aux, st.kmesh, st.nspins, R_CUT)
    for I, K, R, C in inp.lri:
        L.librpa_gpu_set_lri_coeffs(h, I, K, R, C)
    for s, (eig, occ, wfc) in enumerate(inp.ks):
        for k in range(st.nk):
            L.librpa_gpu_set_green(h, s, k, eig[k], occ[k], wfc[k], inp.efermi)
    torch.cuda.synchronize()
    for q in range(st.nk):
        L.librpa_gpu_set_coulomb_dev(h, q, inp.v[q].data_ptr())
    torch.cuda.synchronize()
    if inp.grid is not None:
        g = inp.grid
        L.librpa_gpu_set_grid(h, g["tau"], g["omega"], g["w_omega"], g["gamma"])
    if case["screen"] > 0:
        L.librpa_gpu_set_screening(h, case["screen"])
    return h


def _matrices(case, seed, device):
    """One V and the chi of every frequency (Hermitian, negative) for the no-allocation call."""
    n, nw = case["natoms"], case["ntau"]
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    a = torch.randn((n, n), dtype=torch.complex128, device=device, generator=gen) / math.sqrt(n)
    v = a @ a.conj().T + 0.1 * torch.eye(n, dtype=torch.float64, device=device)
    b = torch.randn((nw, n, n), dtype=torch.complex128, device=device, generator=gen) / math.sqrt(n)
    fall = 1.0 / (0.5 + torch.arange(nw, dtype=torch.float64, device=device))[:, None, None]
    chi = -fall * (b @ b.conj().transpose(1, 2))
    return (0.5 * (v + v.conj().T)).contiguous(), (0.5 * (chi + chi.conj().transpose(1, 2))).contiguous()


def prepare(case, seed):
    s = _State(case)
    if case["call"] == "noalloc":
        s.v, s.chi = _matrices(case, seed, "cuda")
        s.out = torch.empty(case["ntau"], dtype=torch.float64, device="cuda")
        L.librpa_gpu_ec_noalloc(case["natoms"], 0, None, None, None)   # its set-up call
        return s
    for i, st in enumerate(_structures(case)):
        stream = torch.cuda.Stream() if case["call"] == "chi0" else None
        s.handles.append(_handle(case, _Inputs(st, case, seed, i), stream))
        s.keep.append(stream)
    s.st = _structures(case)[0]
    if case["call"] == "batch":
        s.batch = L.librpa_gpu_batch_create(s.handles)
    if case["call"] == "chi0":
        n = s.st.naux
        s.out = torch.empty((s.st.nk, case["ntau"], n, n), dtype=torch.complex128, device="cuda")
    if case["call"] == "ec":
        L.librpa_gpu_chi0(s.handles[0])
    return s


def run(state):
    c = state.case
    if c["call"] == "noalloc":
        L.librpa_gpu_ec_noalloc(c["natoms"], c["ntau"], state.v.data_ptr(), state.chi.data_ptr(), state.out.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
        return state.out
    if c["call"] == "batch":
        return L.librpa_gpu_batch_run(state.batch)
    h, nk = state.handles[0], state.st.nk
    if c["call"] != "ec":
        L.librpa_gpu_chi0(h)
    if c["call"] == "chi0":
        for q in range(nk):
            for w in range(c["ntau"]):
                L.librpa_gpu_get_chi0_freq_dev(h, q, w, state.out[q, w].data_ptr())
        return state.out
    ec, ec_q, ec_w = L.librpa_gpu_ec(h, nk, c["ntau"])
    return {"ec": np.float64(ec), "ec_q": ec_q, "ec_w": ec_w}


# ------------------------------------------------------------------ what a pass cannot do without


@functools.lru_cache(maxsize=256)
def _chi0_flops(st):
    """Flops of Algorithm 1 for one (R, tau) point: the N and X steps, the assembly, the contraction."""
    I, J, R, _ = st.pairs_within(R_CUT)
    m = np.zeros(st.nat)
    np.add.at(m, I, st.n_ao[J])
    union = {(int(j), tuple(r)) for j, r in zip(J, R)}
    m_all = float(sum(st.n_ao[j] for j, _ in union))
    rows = st.n_aux * st.n_ao
    f = 4.0 * float((rows * m).sum()) * (m_all + st.nao)
    f += 8.0 * float((st.n_aux * st.n_ao).sum()) * float((st.n_ao * m).sum())
    return f + 2.0 * st.naux * float((rows * m).sum()), float((rows * m).sum())


def work(case):
    nw = case["ntau"]
    if case["call"] == "noalloc":
        n = case["natoms"]
        return {"bytes": 16.0 * n * n * (nw + 1) + 8.0 * nw, "flops": 8.0 * n ** 3 * (1 / 6 + nw * 2 / 3)}
    flops = nbytes = 0.0
    for st in _structures(case):
        n, nk = float(st.naux), st.nk
        own = sum(q == p for q, p in enumerate(_minus(st.kmesh)))   # q = -q: real matrices
        pair = (nk - own) // 2
        lri = _chi0_flops(st)[1]
        if case["call"] != "ec":
            flops += (own + pair) * nw * _chi0_flops(st)[0] * st.nspins      # chi0(R, tau), R <= -R
            flops += 16.0 * st.nspins * nw * (own + pair) * st.nao ** 3 / 2  # G, k <= -k
            flops += n * n * (2.0 * nk * nw * nw + 4.0 * nk * nw * (own + pair))
            nbytes += 8.0 * lri + 16.0 * st.nspins * nk * st.nao ** 2
        if case["call"] == "chi0":
            nbytes += 16.0 * nk * nw * n * n
        else:
            flops += (2.0 * own + 8.0 * pair) * n ** 3 * (1 / 6 + nw * 2 / 3)
            nbytes += 16.0 * nk * n * n + (16.0 * nk * nw * n * n if case["call"] == "ec" else 0.0)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits


def _exact_chi0(inp, grid):
    """chi0(q, i omega) for q <= -q as a sum over Kohn-Sham states: pair densities of the two-centre
    expansion, weighted with the transform of exp(-Delta tau) over the grid."""
    st, dev = inp.st, inp.v.device
    kf, mi = _kfrac(st.kmesh), _minus(st.kmesh)
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    gamma, tau = to(grid["gamma"]), to(grid["tau"])
    per_atom = [[b for b in inp.lri if b[0] == U] for U in range(st.nat)]
    packed = [to(np.concatenate([b[3] for b in blocks], axis=2)).to(torch.complex128) for blocks in per_atom]
    rows = [np.concatenate([st.off[b[1]] + np.arange(st.n_ao[b[1]]) for b in blocks]) for blocks in per_atom]
    cell = [np.concatenate([np.tile(b[2], (st.n_ao[b[1]], 1)) for b in blocks]) for blocks in per_atom]
    index = {tuple(x): i for i, x in enumerate(itertools.product(*[range(n) for n in st.kmesh]))}
    grid_k = list(index)
    chi = {}
    for q in (x for x in range(st.nk) if x <= mi[x]):
        chi[q] = torch.zeros((len(tau), st.naux, st.naux), dtype=torch.complex128, device=dev)
        for eig, occ, wfc in inp.ks:
            spin = 2.0 if st.nspins == 1 else 1.0
            for k in range(st.nk):
                kq = index[tuple((a + b) % n for a, b, n in zip(grid_k[k], grid_k[q], st.kmesh))]
                no = int((occ[k] > 0).sum())
                co, cv = to(wfc[k][:no].T), to(wfc[kq][no:].T)      # [ao][n], [ao][m]
                rho = torch.empty((st.naux, no, cv.shape[1]), dtype=torch.complex128, device=dev)
                for U in range(st.nat):
                    s = slice(st.off[U], st.off[U + 1])
                    po = to(np.exp(2j * np.pi * (cell[U] @ kf[k])))[:, None] * co[rows[U]]
                    pv = to(np.exp(2j * np.pi * (cell[U] @ kf[kq])))[:, None] * cv[rows[U]]
                    a = torch.einsum("uin,im->unm", packed[U] @ po.conj(), cv[s])
                    b = torch.einsum("uim,in->unm", packed[U] @ pv, co[s].conj())
                    rho[st.xoff[U]:st.xoff[U + 1]] = a + b
                rho = rho.reshape(st.naux, -1)
                delta = to(eig[kq][None, no:] - eig[k][:no, None]).reshape(-1)
                ker = gamma @ torch.exp(-tau[:, None] * delta[None, :])
                real = mi[k] == k and mi[q] == q
                for w in range(len(tau)):
                    if real:
                        r = rho.real
                        chi[q][w] -= (spin / st.nk) * ((r * ker[w]) @ r.T)
                    else:
                        chi[q][w] -= (spin / st.nk) * ((rho * ker[w]) @ rho.conj().T)
    return chi


def _integrand(chi, v):
    p = chi @ v
    one = torch.eye(p.shape[-1], dtype=p.dtype, device=p.device)
    return torch.linalg.slogdet(one - p)[1] + torch.diagonal(p, dim1=-2, dim2=-1).sum(-1).real


def _exact_cost(case):
    f = 0.0
    for st in _structures(case):
        own = sum(q == p for q, p in enumerate(_minus(st.kmesh)))
        per = st.nspins * st.naux ** 2 * float(st.nocc) * (st.nao - st.nocc) * case["ntau"]
        f += st.nk * per * (2.0 * own if own == st.nk else 8.0 * (own + (st.nk - own) / 2))
    return f


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if case["call"] == "noalloc":
        v, chi = _matrices(case, seed, device)
        return _integrand(chi, v)
    # no value under screening (it acts on the real-space Green's functions), on the library's own grid,
    # or where the sum over states takes too long
    if case["screen"] > 0 or _exact_cost(case) > 1.2e13:
        return None
    energies = []
    for i, st in enumerate(_structures(case)):
        inp = _Inputs(st, case, seed, i)
        if inp.grid is None:
            return None
        chi, mi = _exact_chi0(inp, inp.grid), _minus(st.kmesh)
        if case["call"] == "chi0":
            return torch.stack([chi[q] if q in chi else chi[mi[q]].conj() for q in range(st.nk)])
        f = torch.stack([_integrand(chi[min(q, mi[q])], inp.v[min(q, mi[q])]) for q in range(st.nk)]).cpu().numpy()
        part = f * inp.grid["w_omega"][None, :] / (2 * math.pi * st.nk)
        energies.append({"ec": part.sum(), "ec_q": part.sum(1), "ec_w": part.sum(0)})
    return np.array([e["ec"] for e in energies]) if case["call"] == "batch" else energies[0]
