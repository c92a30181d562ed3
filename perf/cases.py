"""Work that users of the engine have it do, as measurable cases.

Every case goes through the public binding (paper_2606_03140_gb300.sedacs), on device arrays as a
program that keeps its state on the GPU calls it.  The kinds:

  md       one XL-BOMD step (sedacs_xlbomd_step): the production loop.  Graph from the previous
           density, halos, Coulomb potential, subgraph densities at 300 K with mu from Eq. 2,
           charges, forces, charge and position update.
  point    energy and forces at a new geometry and given charges: sedacs_graph_build (the cores
           stay), sedacs_subgraph_density with the chemical potential of the geometry before as the
           guess, sedacs_forces, sedacs_energy.  The distance graph is taken at 4 A, which gives the
           subgraph sizes the density graph of an MD run has (about 500 orbitals, 128 to 660).
  scc      two self-consistency iterations with linear mixing in the three-plane bf16 form, which
           the ground state of every run is computed in.
  coulomb  the periodic Coulomb potential alone.
  graph    a new structure: atom graph, cores, halos, and the lists read back.
  gnn      the learned charge-response kernel: one application and one parameter gradient.

The engine's FP32-class forms (precision 1 to 4) compute in FP32-class arithmetic, whatever the width
of the arrays at its boundary; their results are handed on in single precision, the FP64 form's in
double precision.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2606_03140_gb300 import inputs as I
from paper_2606_03140_gb300 import sedacs as S

DEV = "cuda"
BOHR = 0.529177210903              # Angstrom
KB = 3.166811563e-6                # Hartree / K
TE = 300.0
V_WATER, V_METHANOL = 29.97, 62.42   # Angstrom^3 per molecule: the densities of the benchmark boxes
R_GRAPH = 4.0                      # Angstrom, distance graph of the point cases
# mean charges (e) of the SCC ground states, by atom of the molecule templates below
Q_WATER = (0.314, -0.157, -0.157)
Q_METHANOL = (-0.04, 0.29, -0.03, -0.03, -0.03, -0.16)


# ---------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest box of the tests, in dynamics: launch and synchronisation latency
        {"name": "md_water96", "kind": "md", "waters": 32, "methanols": 0, "precision": 1},
        # the benchmark's box: one production step
        {"name": "md_water9000", "kind": "md", "waters": 3000, "methanols": 0, "precision": 1},
        # energies and forces from the smallest box to the largest the repository runs
        {"name": "point_water96", "kind": "point", "waters": 32, "methanols": 0, "precision": 1},
        {"name": "point_water1533", "kind": "point", "waters": 511, "methanols": 0, "precision": 1},
        # the liquid mixture: three species, ragged subgraphs
        {"name": "point_mix2997", "kind": "point", "waters": 333, "methanols": 333, "precision": 1},
        {"name": "point_water9000", "kind": "point", "waters": 3000, "methanols": 0, "precision": 1},
        {"name": "point_water30000", "kind": "point", "waters": 10000, "methanols": 0, "precision": 1},
        # the ground-state iterations before a run (three bf16 planes in every product)
        {"name": "scc_water1533", "kind": "scc", "waters": 511, "methanols": 0, "precision": 4},
        # the plain FP64 form, which a user checks the others with on small boxes
        {"name": "point_fp64_water288", "kind": "point", "waters": 96, "methanols": 0, "precision": 0},
        # the Coulomb sums alone at the largest size
        {"name": "coulomb_water30000", "kind": "coulomb", "waters": 10000, "methanols": 0, "precision": 1},
        # graph, cores and halos of a new structure
        {"name": "graph_water9000", "kind": "graph", "waters": 3000, "methanols": 0, "precision": 1},
        # the learned kernel on the benchmark's box
        {"name": "gnn_water9000", "kind": "gnn", "waters": 3000, "methanols": 0, "precision": 1},
    ]


# the most molecules a drawn case of each kind has
_MOST = {"md": 3000, "point": 3000, "scc": 700, "fp64": 96, "coulomb": 10000, "graph": 10000, "gnn": 3000}


def draw(rng):
    kind = rng.choice(["md", "md", "md", "point", "point", "point", "point", "scc", "fp64", "coulomb", "graph", "gnn"])
    mols = round(math.exp(rng.uniform(math.log(32), math.log(_MOST[kind]))))
    # a third of the boxes are mixtures; a methanol counts as two waters (six atoms, twelve orbitals)
    methanols = round(mols * rng.uniform(0.05, 0.5) / 2) if rng.random() < 1 / 3 else 0
    precision = {"scc": 4, "fp64": 0}.get(kind, 1)
    return {"kind": "point" if kind == "fp64" else kind, "waters": mols - 2 * methanols, "methanols": methanols,
            "precision": precision}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _template(kind):
    """Atoms of one molecule: species, positions about the centre (Angstrom), charges."""
    if kind == 0:
        half = math.radians(104.5) / 2
        pos = 0.96 * np.array([[0, 0, 0], [math.sin(half), 0, math.cos(half)], [-math.sin(half), 0, math.cos(half)]])
        sp, q = (I.O, I.H, I.H), Q_WATER
    else:
        tet, ang = math.acos(-1 / 3), math.radians(71.5)
        h = [(1.09 * math.sin(tet) * math.cos(2 * math.pi * k / 3), 1.09 * math.sin(tet) * math.sin(2 * math.pi * k / 3),
              1.09 * math.cos(tet)) for k in range(3)]
        pos = np.array([(0, 0, 0), (0, 0, 1.43), *h, (-0.96 * math.sin(ang), 0, 1.43 + 0.96 * math.cos(ang))])
        sp, q = (I.C, I.O, I.H, I.H, I.H, I.H), Q_METHANOL
    return sp, pos - pos.mean(axis=0), q


def _rotations(rng, m):
    q = rng.standard_normal((m, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.stack([np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)], 1),
                     np.stack([2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)], 1),
                     np.stack([2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1)], 1)


def _inputs(case, seed):
    """A liquid box: molecules on fcc sites with jitter and random orientations, no two molecules closer
    than 1.2 Angstrom where 100 redraws can avoid it; charges near the ground state's; velocities at 300 K."""
    rng = np.random.default_rng([seed, case["waters"], case["methanols"]])
    nw, nm = case["waters"], case["methanols"]
    n_mol = nw + nm
    box = np.full(3, (V_WATER * nw + V_METHANOL * nm) ** (1 / 3))
    m = math.ceil((n_mol / 4) ** (1 / 3) - 1e-12)
    grid = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
    sites = ((grid + np.array([[0, 0, 0], [.5, .5, 0], [.5, 0, .5], [0, .5, .5]])).reshape(-1, 3) + 0.25) * (box / m)
    sites = sites[np.sort(rng.choice(len(sites), n_mol, replace=False))] + rng.uniform(-0.2, 0.2, (n_mol, 3))
    kinds = rng.permutation(np.repeat([0, 1], [nw, nm]))
    tem = [_template(0), _template(1)]
    size = np.array([3, 6])[kinds]
    first = np.concatenate([[0], np.cumsum(size)])
    mol = np.repeat(np.arange(n_mol), size)
    species = np.concatenate([tem[k][0] for k in kinds]).astype(np.int32)
    charge = np.concatenate([tem[k][2] for k in kinds])
    body = np.concatenate([tem[k][1] for k in kinds])
    R = np.zeros((first[-1], 3))
    redo = np.arange(n_mol)
    bt, mt = torch.tensor(box, device=DEV), torch.tensor(mol, device=DEV)
    Rt = torch.zeros(R.shape, dtype=torch.float64, device=DEV)
    for _ in range(100):
        rot = np.zeros((n_mol, 3, 3))
        rot[redo] = _rotations(rng, len(redo))
        at = np.nonzero(np.isin(mol, redo))[0]
        R[at] = sites[mol[at]] + np.einsum("aij,aj->ai", rot[mol[at]], body[at])
        Rt[torch.tensor(at, device=DEV)] = torch.tensor(R[at], device=DEV)
        close = torch.zeros(n_mol, dtype=torch.bool, device=DEV)
        for a in torch.tensor(at, device=DEV).split(2048):
            d = Rt[None, :, :] - Rt[a, None, :]
            d -= bt * torch.round(d / bt)
            hit = ((d * d).sum(-1) < 1.2**2) & (mt[None, :] != mt[a, None])
            close[mt[a[hit.any(1)]]] = True
        redo = np.nonzero(close.cpu().numpy())[0]
        if len(redo) == 0:
            break
    n = charge + 0.01 * rng.standard_normal(len(R))
    n -= n.mean()
    V = I.maxwell_boltzmann(species, 300.0, int(rng.integers(1 << 30)))
    return species, box, R, n, V


@functools.lru_cache(maxsize=1)
def _model():
    return I.default_model()


class _State:
    """A context on the current stream, the arrays the program keeps on the GPU, and its results' type."""

    def __init__(self, case, seed, **params):
        self.case = case
        self.species, self.box, R, n, V = _inputs(case, seed)
        self.N = len(R)
        self.R, self.n, self.V = (torch.tensor(x, device=DEV) for x in (R, n, V))
        self.dtype = torch.float64 if case["precision"] == 0 else torch.float32
        self.params = S.sedacs_default_params(precision=case["precision"], **params)
        self.ctx = S.sedacs_create(self.species, self.box, _model(), self.params)
        torch.cuda.synchronize()
        S.sedacs_set_device_io(self.ctx, True, torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        if getattr(self, "ctx", None):
            S.sedacs_destroy(self.ctx)
            self.ctx = None

    def out(self, x):
        return x.to(self.dtype) if isinstance(x, torch.Tensor) else torch.tensor(x, dtype=self.dtype)


def _settle(s):
    """Twelve iterations of linear mixing: what is left is the slow tail of the ground-state search."""
    S.sedacs_graph_build(s.ctx, s.R)
    S.sedacs_partition(s.ctx, s.R)
    mu, _, _, _ = S.sedacs_scc_step(s.ctx, s.R, s.n, max_iter=12)
    return mu


def prepare(case, seed):
    kind = case["kind"]
    if kind == "md":
        # the state of a run: near-ground-state charges, cores, and two steps for mu's extrapolation
        s = _State(case, seed, c_k0=0.05)
        mu = _settle(s)
        S.sedacs_xlbomd_init(s.ctx, s.R, s.V, s.n, mu)
        s.E = torch.zeros((1, 3), dtype=torch.float64, device=DEV)
        s.n_out = torch.zeros_like(s.n)
        for _ in range(2):
            S.sedacs_xlbomd_step(s.ctx, s.R, s.V, 1, 0.25, s.E, s.n_out)
    elif kind == "scc":
        s = _State(case, seed)
        s.mu = _settle(s)
    elif kind == "point":
        # the cores, and the chemical potential of the geometry one time step before
        s = _State(case, seed, r_graph=R_GRAPH)
        before = s.R - 0.25 * s.V
        S.sedacs_graph_build(s.ctx, before)
        S.sedacs_partition(s.ctx, before)
        s.q, s.F = torch.zeros_like(s.n), torch.zeros_like(s.R)
        s.mu, _, _, _ = S.sedacs_subgraph_density(s.ctx, before, s.n, q=s.q)
    elif kind == "coulomb":
        s = _State(case, seed)
        s.pot = torch.zeros_like(s.n)
    elif kind == "graph":
        s = _State(case, seed, r_graph=R_GRAPH)
        # the program's own lists, with room for every structure of this size
        s.col, s.sub_atoms = np.zeros(48 * s.N, np.int32), np.zeros(24 * s.N + 4096, np.int32)
    else:
        s = _State(case, seed, r_graph=R_GRAPH)
        S.sedacs_graph_build(s.ctx, s.R)
        p, s.y, s.gu = _gnn_inputs(case, seed, s.N)
        S.sedacs_gnn_set_params(s.ctx, p)
    return s


def _gnn_inputs(case, seed, N):
    """Network parameters as sedacs_gnn_init draws them (scaled normals), a residual and a weight vector."""
    rng = np.random.default_rng([seed, 77])
    layer = [0.1 * rng.standard_normal(8 * 64), 0.0125 * rng.standard_normal(2 * 64 * 64)]
    p = np.concatenate([0.1 * rng.standard_normal(192), *layer, *[-x for x in layer], *[x[::-1] for x in layer],
                        0.1 * rng.standard_normal(64)])
    return p, 0.01 * rng.standard_normal(N), rng.standard_normal(N)


def run(s):
    kind = s.case["kind"]
    if kind == "md":
        S.sedacs_xlbomd_step(s.ctx, s.R, s.V, 1, 0.25, s.E, s.n_out)
        return {"R": s.out(s.R), "V": s.out(s.V), "E": s.out(s.E), "n": s.out(s.n_out)}
    if kind == "point":
        S.sedacs_graph_build(s.ctx, s.R)
        # (mu itself is no result: in a gap the electron count leaves it open)
        _, q, _, _ = S.sedacs_subgraph_density(s.ctx, s.R, s.n, s.mu, q=s.q)
        F = S.sedacs_forces(s.ctx, s.N, F=s.F)
        e = S.sedacs_energy(s.ctx)
        return {"q": s.out(q), "F": s.out(F), "e": s.out(torch.from_numpy(e))}
    if kind == "scc":
        n = s.n.clone()
        _, residual, _, _ = S.sedacs_scc_step(s.ctx, s.R, n, max_iter=2, mu=s.mu)
        return {"n": s.out(n), "residual": s.out(residual)}
    if kind == "coulomb":
        return s.out(S.sedacs_coulomb_potential(s.ctx, s.R, s.n, V=s.pot))
    if kind == "graph":
        nnz = S.sedacs_graph_build(s.ctx, s.R)
        S.sedacs_partition(s.ctx, s.R)
        ptr, col = S.sedacs_graph_get(s.ctx, s.N, nnz)
        sub_ptr, sub_atoms, n_core = S.sedacs_parts_get(s.ctx)
        for own, new in ((s.col, col), (s.sub_atoms, sub_atoms)):
            own[:len(new)], own[len(new):] = new, -1
        return {"ptr": ptr, "col": s.col, "sub_ptr": sub_ptr, "sub_atoms": s.sub_atoms, "n_core": n_core}
    return {"u": s.out(torch.from_numpy(S.sedacs_gnn_apply(s.ctx, s.y))),
            "grad": s.out(torch.from_numpy(S.sedacs_gnn_param_grad(s.ctx, s.y, s.gu)))}


# ---------------------------------------------------------------------------------------------
# the work that cannot be done without
# ---------------------------------------------------------------------------------------------
def work(case):
    nw, nm = case["waters"], case["methanols"]
    N = 3 * nw + 6 * nm
    vol = V_WATER * nw + V_METHANOL * nm
    orbs = 6 * nw + 12 * nm
    kind = case["kind"]
    io = 8.0 * N * {"md": 14, "point": 8, "scc": 5, "coulomb": 5, "graph": 3, "gnn": 3}[kind]
    edges = N * N / vol * 4 / 3 * math.pi * R_GRAPH**3
    if kind == "graph":
        return {"bytes": io + 4 * edges + 8 * N, "flops": 10 * edges}
    if kind == "gnn":
        # per layer: the radial filter and the message of every edge, two 64 x 64 mixes of every atom;
        # forward, and a backward pass of twice its work
        return {"bytes": io + 36 * edges, "flops": 3 * 3 * (2 * 64 * 9 * edges + 4 * 64 * 64 * N)}
    # Coulomb sums: pairs within 15 A (or half the box) at about 40 operations, and the reciprocal part
    coul = N * 40 * N / vol * 4 / 3 * math.pi * min(15.0, vol ** (1 / 3) / 2) ** 3 * 2
    if kind == "coulomb":
        return {"bytes": io, "flops": coul}
    # subgraphs: a core of 32 atoms with everything within 4 A of it
    parts = max(1, round(N / 32))
    a, r = (vol / parts) ** (1 / 3), R_GRAPH
    n = orbs / vol * min(vol, a**3 + 6 * a * a * r + 3 * math.pi * a * r * r + 4 / 3 * math.pi * r**3)
    # symmetric products of n^3: three for S^-1/2, three for h~, fifteen for a Fermi operator whose
    # polynomial has a degree of at least 2^15 at 300 K, and the core rows of the density matrix
    evals = 2 if kind == "scc" else 1
    return {"bytes": io, "flops": parts * evals * (21 * n**3 + 8 * n * n * orbs / parts) + coul * evals}


# ---------------------------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------------------------
def _min_image(R, i, j, box):
    d = R[j] - R[i]
    return d - box * torch.round(d / box)


def _shifts(box, r_cut):
    k = [range(-int((r_cut + 0.5 * b) // b), int((r_cut + 0.5 * b) // b) + 1) for b in box]
    k = torch.tensor([[x, y, z] for x in k[0] for y in k[1] for z in k[2]], dtype=torch.float64, device=DEV)
    return k * torch.tensor(box, device=DEV)


def _pairs(R, box, r_cut):
    """(i, j, R_j - R_i + L) of every pair and image closer than r_cut, but an atom with itself."""
    bt, found = torch.tensor(box, device=DEV), []
    for L in _shifts(box, r_cut):
        for i in torch.arange(len(R), device=DEV).split(max(1, (1 << 24) // len(R))):
            d = R[None, :, :] - R[i, None, :]
            d = d - bt * torch.round(d / bt) + L
            r2 = (d * d).sum(-1)
            a, b = torch.nonzero((r2 < r_cut * r_cut) & (r2 > 0), as_tuple=True)
            found.append((i[a], b, d[a, b]))
    return [torch.cat(x) for x in zip(*found)]


def _coulomb(R_A, species, box, b, a=None):
    """V = gamma b by Ewald sums to 1e-13; with a, also the gradient of a^T gamma b (Ha / Angstrom)."""
    R, L = R_A / BOHR, np.asarray(box) / BOHR
    u = torch.tensor(_model().hubbard_u, dtype=torch.float64, device=DEV)[species]
    sig2 = 1 / (math.pi * u * u)
    x = math.sqrt(-math.log(1e-13))
    rc = min(12.0, max(8.0, 0.45 * min(box))) / BOHR
    eta = (x + 0.3) / rc
    kmax, vol, tp = 2 * eta * x, float(np.prod(L)), 2 / math.sqrt(math.pi)
    V = -math.pi / (eta * eta * vol) * b.sum() + (u - eta * tp) * b
    G = torch.zeros_like(R)
    bt = torch.tensor(L, device=DEV)
    for sh in _shifts(L, rc):
        for i in torch.arange(len(R), device=DEV).split(max(1, (1 << 24) // len(R))):
            dv = R[None, :, :] - R[i, None, :]
            dv = dv - bt * torch.round(dv / bt) + sh
            d = dv.norm(dim=-1)
            ii, jj = torch.nonzero((d < rc) & (d > 0), as_tuple=True)
            d, dv = d[ii, jj], dv[ii, jj]
            I_ = i[ii]
            s = 1 / torch.sqrt(2 * (sig2[I_] + sig2[jj]))
            phi = (torch.erfc(eta * d) - torch.erfc(s * d)) / d
            V.index_add_(0, I_, phi * b[jj])
            if a is not None:
                dphi = tp * (s * torch.exp(-(s * d) ** 2) - eta * torch.exp(-(eta * d) ** 2)) / d - phi / d
                G.index_add_(0, I_, (-(a[I_] * b[jj] + a[jj] * b[I_]) * dphi / d)[:, None] * dv)
    nmax = [int(kmax * l / (2 * math.pi)) for l in L]
    m = torch.cartesian_prod(*[torch.arange(-k, k + 1, device=DEV) for k in nmax]).double()
    k = m * (2 * math.pi / bt)
    k2 = (k * k).sum(1)
    half = (m[:, 0] > 0) | ((m[:, 0] == 0) & ((m[:, 1] > 0) | ((m[:, 1] == 0) & (m[:, 2] > 0))))
    k, k2 = k[half & (k2 <= kmax * kmax)], k2[half & (k2 <= kmax * kmax)]
    w = 8 * math.pi / vol * torch.exp(-k2 / (4 * eta * eta)) / k2
    for kk, ww in zip(k.split(max(64, (1 << 25) // len(R))), w.split(max(64, (1 << 25) // len(R)))):
        ph = R @ kk.T
        c, s = torch.cos(ph), torch.sin(ph)
        bc, bs = ww * (b @ c), ww * (b @ s)
        V += c @ bc + s @ bs
        if a is not None:
            ac, as_ = ww * (a @ c), ww * (a @ s)
            G += (a[:, None] * (c * bs - s * bc) + b[:, None] * (c * as_ - s * ac)) @ kk
    return V, G / BOHR


def _blocks(d, si, sj):
    """4 x 4 Slater-Koster blocks (s, px, py, pz) at the displacements d; the overlap is a multiple of them."""
    m = _model()
    v0 = torch.tensor(m.v0, dtype=torch.float64, device=DEV)
    r = d.norm(dim=-1)
    l = d / r[:, None]
    t = ((r - m.r_on) / (m.r_off - m.r_on)).clamp(0, 1)
    g = torch.exp(-r / m.decay) * (1 - 10 * t**3 + 15 * t**4 - 6 * t**5)
    ss, sp, ps = v0[si, sj, 0] * g, v0[si, sj, 1] * g, v0[sj, si, 1] * g
    pps, ppp = v0[si, sj, 2] * g, v0[si, sj, 3] * g
    pp = l[:, :, None] * l[:, None, :] * (pps - ppp)[:, None, None] + ppp[:, None, None] * torch.eye(3, device=DEV)
    top = torch.cat([ss[:, None], l * sp[:, None]], 1)[:, None, :]
    return torch.cat([top, torch.cat([-(l * ps[:, None])[:, :, None], pp], 2)], 1)


def _graph(R, box, r_cut):
    """Sorted CSR of the atoms closer than r_cut (minimum image)."""
    bt, rows, cols = torch.tensor(box, device=DEV), [], []
    for i in torch.arange(len(R), device=DEV).split(max(1, (1 << 24) // len(R))):
        d = R[None, :, :] - R[i, None, :]
        d = d - bt * torch.round(d / bt)
        near = ((d * d).sum(-1) < r_cut * r_cut) & (torch.arange(len(R), device=DEV) != i[:, None])
        a, b = torch.nonzero(near, as_tuple=True)
        rows.append(i[a])
        cols.append(b)
    row, col = torch.cat(rows).cpu().numpy(), torch.cat(cols).cpu().numpy()
    return np.concatenate([[0], np.cumsum(np.bincount(row, minlength=len(R)))]), col


def _cores(R, box, size):
    """Recursive bisection along the widest axis, by (wrapped coordinate, index); each core ascending."""
    w = R - box * np.floor(R / box)
    out, todo = [], [(np.arange(len(R)), max(1, int(np.rint(len(R) / size))))]
    while todo:
        at, p = todo.pop()
        if p == 1:
            out.append(np.sort(at))
            continue
        ax = int(np.argmax(w[at].max(0) - w[at].min(0)))
        at = at[np.lexsort((at, w[at, ax]))]
        cut = len(at) * (p // 2) // p
        todo += [(at[cut:], p - p // 2), (at[:cut], p // 2)]
    return out


def _subgraphs(ptr, col, cores, N):
    out = []
    for c in cores:
        near = np.zeros(N, bool)
        near[np.concatenate([col[ptr[a]:ptr[a + 1]] for a in c])] = True
        near[c] = False
        out.append((np.concatenate([c, np.nonzero(near)[0]]), len(c)))
    return out


def _point(case, seed):
    m = _model()
    species, box, R_h, n_h, vel = _inputs(case, seed)
    R, n = torch.tensor(R_h, device=DEV), torch.tensor(n_h, device=DEV)
    sp = torch.tensor(species, device=DEV).long()
    before = R_h - 0.25 * vel          # the cores were made there
    N = len(R)
    V, _ = _coulomb(R, sp, box, n)
    subs = _subgraphs(*_graph(R, box, R_GRAPH), _cores(before, box, 32), N)
    pi, pj, pd = _pairs(R, box, m.r_off)
    blocks = _blocks(pd, sp[pi], sp[pj])
    order = torch.argsort(pi, stable=True)
    pi, pj, pd, blocks = pi[order], pj[order], pd[order], blocks[order]
    start = torch.searchsorted(pi, torch.arange(N + 1, device=DEV))
    norb = np.asarray(m.n_orb)[species]
    eps = np.stack([np.asarray(m.eps_s)[species]] + [np.asarray(m.eps_p)[species]] * 3, 1)
    solved = []
    for atoms, nc in subs:
        at = torch.tensor(atoms, device=DEV)
        local = torch.full((N,), -1, device=DEV)
        local[at] = torch.arange(len(at), device=DEV)
        spans = zip(start[at].tolist(), start[at + 1].tolist())
        take = torch.cat([torch.arange(a, b, device=DEV) for a, b in spans])
        take = take[local[pj[take]] >= 0]
        i, j = local[pi[take]], local[pj[take]]
        H4 = torch.zeros((len(at), len(at), 4, 4), dtype=torch.float64, device=DEV)
        H4.index_put_((i, j), blocks[take], accumulate=True)
        keep = np.nonzero((np.arange(4)[None, :] < norb[atoms][:, None]).ravel())[0]
        B = H4.permute(0, 2, 1, 3).reshape(4 * len(at), 4 * len(at))
        kt = torch.tensor(keep, device=DEV)
        B = B[kt][:, kt].cpu().numpy()
        s = m.overlap_scale * B + np.eye(len(B))
        v = np.repeat(V.cpu().numpy()[atoms], norb[atoms])
        h = B + np.diag(eps[atoms].ravel()[keep]) + 0.5 * s * (v[:, None] + v[None, :])
        lam, X = np.linalg.eigh(s)
        Z = (X / np.sqrt(lam)) @ X.T
        e, X = np.linalg.eigh(Z @ h @ Z)
        C = Z @ X
        nco = int(norb[atoms[:nc]].sum())
        weight = np.sum(C[:nco] * (s[:nco] @ C), axis=0)
        solved.append((atoms, nc, nco, s, C, e, weight, B + np.diag(eps[atoms].ravel()[keep]), take, keep))
    beta = 1 / (KB * TE)
    f = lambda x: 0.5 * (1 - np.tanh(0.5 * beta * x))  # noqa: E731
    allE, allW = np.concatenate([x[5] for x in solved]), np.concatenate([x[6] for x in solved])
    ne = float(np.asarray(m.z_val)[species].sum())
    lo, hi = allE.min() - 1, allE.max() + 1
    for _ in range(90):
        mu = 0.5 * (lo + hi)
        lo, hi = (mu, hi) if 2 * float(allW @ f(allE - mu)) < ne else (lo, mu)
    q, band = -np.asarray(m.z_val)[species].astype(float), 0.0
    dU = torch.zeros_like(R)
    for atoms, nc, nco, s, C, e, _, h0, take, keep in solved:
        occ = f(e - mu)
        D, W = 2 * (C[:nco] * occ) @ C.T, 2 * (C[:nco] * (occ * e)) @ C.T
        pop = np.sum(D * s[:nco], axis=1)
        band += float(np.sum(D * h0[:nco]))
        q[atoms[:nc]] += np.add.reduceat(pop, np.concatenate([[0], np.cumsum(norb[atoms[:nc]])[:-1]]))
        # forces: the blocks' derivatives contracted with D (1 + S-scale of the shift) and W
        at = torch.tensor(atoms, device=DEV)
        local = torch.full((N,), -1, device=DEV)
        local[at] = torch.arange(len(at), device=DEV)
        core = local[pi[take]] < nc
        t = take[core]
        full = np.zeros((2, 4 * nc, 4 * len(atoms)))
        full[:, keep[:nco, None], keep[None, :]] = np.stack([D, W])
        full = torch.tensor(full, device=DEV).reshape(2, nc, 4, len(atoms), 4)
        i, j = local[pi[t]], local[pj[t]]
        Db, Wb = full[0, i, :, j, :], full[1, i, :, j, :]
        M = Db + m.overlap_scale * (0.5 * (V[pi[t]] + V[pj[t]])[:, None, None] * Db - Wb)
        d = pd[t].clone().requires_grad_()
        (M * _blocks(d, sp[pi[t]], sp[pj[t]])).sum().backward()
        dU.index_add_(0, pj[t], d.grad)
        dU.index_add_(0, pi[t], -d.grad)
    qt = torch.tensor(q, device=DEV)
    _, G = _coulomb(R, sp, box, n, qt - 0.5 * n)
    amp = torch.tensor(m.rep_array(), device=DEV)[sp[pi], sp[pj]]
    d = pd.clone().requires_grad_()
    r = d.norm(dim=-1)
    t = ((r - m.r_on) / (m.r_off - m.r_on)).clamp(0, 1)
    rep = (0.5 * amp * torch.exp(-r / m.rep_decay) * (1 - 10 * t**3 + 15 * t**4 - 6 * t**5)).sum()
    rep.backward()
    dU.index_add_(0, pj, d.grad)
    dU.index_add_(0, pi, -d.grad)
    coul, rep = float((qt - 0.5 * n) @ V), float(rep)
    return {"q": qt, "F": -(dU + G),
            "e": torch.tensor([band, coul, rep, band + coul + rep], dtype=torch.float64)}


def _gnn(case, seed):
    species, box, R_h, _, _ = _inputs(case, seed)
    R = torch.tensor(R_h, device=DEV)
    N = len(R)
    p, y, gu = (torch.tensor(x, device=DEV) for x in _gnn_inputs(case, seed, N))
    p.requires_grad_()
    ptr, col = _graph(R, box, R_GRAPH)
    i, j = torch.tensor(np.repeat(np.arange(N), np.diff(ptr)), device=DEV), torch.tensor(col, device=DEV)
    r = _min_image(R, i, j, torch.tensor(box, device=DEV)).norm(dim=-1)
    centre = torch.linspace(0.8, 6.0, 8, dtype=torch.float64, device=DEV)
    basis = torch.exp(-(((r[:, None] - centre) / 0.7) ** 2)) * (0.5 * (torch.cos(math.pi * r / 6) + 1) * (r < 6))[:, None]
    h = y[:, None] * p[:192].reshape(3, 64)[torch.tensor(species, device=DEV).long()]
    o = 192
    for _ in range(3):
        C, A, B = p[o:o + 512].reshape(8, 64), p[o + 512:o + 4608].reshape(64, 64), p[o + 4608:o + 8704].reshape(64, 64)
        o += 8704
        a = torch.zeros_like(h).index_add(0, i, (basis @ C) * h[j])
        h = h + a @ A.T + h @ B.T
    u = -0.5 * y + h @ p[o:]
    (gu * u).sum().backward()
    return {"u": u.detach(), "grad": p.grad}


def exact(case, seed):
    """None for what a trajectory or an iteration returns (it depends on the density graph's threshold) and for
    whole numbers; the largest box would take too long."""
    if case["kind"] == "point" and case["waters"] + 2 * case["methanols"] <= 3000:
        return _point(case, seed)
    if case["kind"] == "coulomb":
        species, box, R, n, _ = _inputs(case, seed)
        sp = torch.tensor(species, device=DEV).long()
        return _coulomb(torch.tensor(R, device=DEV), sp, box, torch.tensor(n, device=DEV))[0]
    if case["kind"] == "gnn":
        return _gnn(case, seed)
    return None
