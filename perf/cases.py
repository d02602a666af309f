"""Performance cases of the exchange build: the calls of an SCF program over their real range.

Every case is what a program that uses the library does again and again with a context
that it keeps: the K build and E_x of an SCF iteration (one density or two spin channels, a
difference density, with or without the Bloch sums of a periodic system), the gradients of a
relaxation step, and the RI fit of a new geometry.  Geometries, species sizes, cutoffs and
densities are the workloads of ``rix_inputs`` (water clusters, ice-like and perovskite-like cells)
at sizes from two molecules to 192 atoms; C and V are drawn on the GPU with the same definitions
(C ~ N(0,1) exp(-0.8 r), V the short-range Coulomb interaction of s-Gaussians).

``exact`` evaluates the same contractions in plain torch FP64, one atom pair at a time, from the
packed inputs and the pair list alone.
"""
import dataclasses
import functools
import json
import math

import numpy as np
import torch

import rix_inputs as ri
from paper_2403_10343_gb300 import rix
from paper_2403_10343_gb300.rix import Exchange

DEV = "cuda"
FIT_LAMBDA = 1e-3  # Tikhonov shift of the fitted metric (the workloads' aux sets are near-singular)


# ---------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: two molecules, every launch counts
        dict(name="dimer_fp64", task="scf", system="cluster", n=2, geom=0, precision="fp64"),
        # a small molecule cluster without cutoff, the accurate and the fast path
        dict(name="cluster8_fp64", task="scf", system="cluster", n=8, geom=0, precision="fp64"),
        dict(name="cluster8_mixed", task="scf", system="cluster", n=8, geom=0, precision="mixed"),
        # an ordinary spin-polarised cluster, an odd number of molecules: two builds per iteration
        dict(name="cluster27_spin_mixed", task="spin", system="cluster", n=27, geom=0, precision="mixed"),
        # the 192-atom cluster with the 8 A cutoff: the ordinary SCF iteration of a larger cluster
        dict(name="cluster64_mixed", task="scf", system="cluster", n=64, geom=1, precision="mixed"),
        dict(name="cluster64_fp64", task="scf", system="cluster", n=64, geom=1, precision="fp64"),
        # a late SCF iteration, K updated from a difference density of which little is left
        dict(name="cluster64_delta_mixed", task="delta", system="cluster", n=64, geom=1, precision="mixed"),
        # a small periodic cell whose atoms meet their own images, with K(k) on a few k points
        dict(name="ice8_fp64_k4", task="scf", system="ice", nx=1, ny=1, nz=1, geom=2, precision="fp64", nk=4),
        # a 192-atom periodic cell: the largest SCF iteration here
        dict(name="ice64_mixed_k2", task="scf", system="ice", nx=2, ny=2, nz=2, geom=2, precision="mixed", nk=2),
        # heavy species (39/140 and 32/120 functions per atom) beside light ones
        dict(name="perovskite12_mixed", task="scf", system="perovskite", nx=1, ny=1, nz=1, geom=3, precision="mixed"),
        # a relaxation step of a cluster: the adjoint and the forces
        dict(name="cluster20_gradient_fp64", task="gradient", system="cluster", n=20, geom=0, precision="fp64"),
        # a new geometry: RI coefficients from the three-centre integrals, loaded into the context
        dict(name="cluster27_fit", task="fit", system="cluster", n=27, geom=0, precision="fp64"),
    ]


def draw(rng):
    geom = rng.randrange(1000)
    precision = rng.choice(["fp64", "mixed"])

    def molecules(lo, hi):
        return min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49))))))

    kind = rng.choice(["cluster", "cluster", "spin", "delta", "ice", "perovskite", "gradient", "fit"])
    if kind == "cluster":
        return dict(task="scf", system="cluster", n=molecules(2, 64), geom=geom, precision=precision)
    if kind in ("spin", "delta"):
        return dict(task=kind, system="cluster", n=molecules(2, 40), geom=geom, precision=precision)
    if kind == "ice":
        nx, ny, nz = rng.choice([(1, 1, 1), (2, 1, 1), (1, 1, 2), (3, 1, 1), (2, 2, 1), (2, 1, 2), (2, 2, 2)])
        if precision == "fp64" and nx * ny * nz > 2:
            precision = "mixed"
        return dict(task="scf", system="ice", nx=nx, ny=ny, nz=nz, geom=geom, precision=precision,
                    nk=rng.randint(0, 4))
    if kind == "perovskite":
        return dict(task="scf", system="perovskite", nx=1, ny=1, nz=1, geom=geom, precision="mixed",
                    nk=rng.randint(0, 4))
    if kind == "gradient":
        return dict(task="gradient", system="cluster", n=molecules(2, 20), geom=geom, precision=precision)
    return dict(task="fit", system="cluster", n=molecules(2, 40), geom=geom, precision="fp64")


# ---------------------------------------------------------------------------- geometry
@functools.lru_cache(maxsize=64)
def _topology(key):
    """System and pair list of a case (the geometry a program has in hand, the same for every seed)."""
    c = json.loads(key)
    if c["system"] == "cluster":
        side = math.ceil(round(c["n"] ** (1.0 / 3.0), 9))
        s = ri.water_cluster(side, c["geom"], cutoff=c["n"] > 8)
        na = 3 * c["n"]
        s = dataclasses.replace(s, name=f"(H2O)_{c['n']}", xyz=s.xyz[:na], species=s.species[:na],
                                orbital_centres=s.orbital_centres[:5 * c["n"]])
    elif c["system"] == "ice":
        s = ri.ice(c["nx"], c["ny"], c["nz"], c["geom"])
    else:
        s = ri.perovskite(c["nx"], c["ny"], c["nz"], c["geom"])
    return s, ri.pair_list(s)


def _packed(case, seed=None):
    c = {k: case[k] for k in ("system", "n", "nx", "ny", "nz", "geom") if k in case}
    s, (keys, A, B, n) = _topology(json.dumps(c, sort_keys=True))
    if seed is not None:  # other draws of C and D; the aux widths too are the seed's
        rng = np.random.default_rng(seed)
        sigma = [np.sort(0.3 * 10.0 ** rng.random(len(w))) for w in s.sigma]
        s = dataclasses.replace(s, seed=int(seed), sigma=sigma)
    return ri.Packed(s, keys, A, B, n)


def _weights(case, pk):
    """Occupations of the localised orbitals, one set per density of the case."""
    m = np.arange(len(pk.system.orbital_centres))
    if case["task"] == "spin":  # the down channel leaves every fifth orbital empty
        return [np.ones(len(m)), np.where(m % 5 == 4, 0.0, 1.0)]
    if case["task"] == "delta":  # an eighth of the orbitals still changes, by a small amount
        return [np.where(m % 8 == 3, 2e-3, 0.0)]
    return [np.full(len(m), 2.0)]


# ---------------------------------------------------------------------------- inputs
def _groups(pk):
    """Representative pairs by (species of A, species of B, on-site)."""
    sp = pk.system.species
    idx = np.nonzero(pk.rep)[0]
    code = (sp[pk.A[idx]].astype(np.int64) * 64 + sp[pk.B[idx]]) * 2 + pk.onsite[idx]
    for g in np.unique(code):
        sel = idx[code == g]
        yield int(sp[pk.A[sel[0]]]), int(sp[pk.B[sel[0]]]), bool(pk.onsite[sel[0]]), sel


def _put(dst, off, sel, blocks):
    """dst[off[p] ...] = blocks[p] for the pairs sel (equal block sizes)."""
    flat = blocks.reshape(len(sel), -1)
    start = torch.as_tensor(off[sel], device=DEV)
    dst[(start[:, None] + torch.arange(flat.shape[1], device=DEV)).reshape(-1)] = flat.reshape(-1)


def _symmetric_C(pk, gen):
    """N(0,1) exp(-0.8 r) in the packed C layout, pair-symmetric bit for bit."""
    s = pk.system
    out = torch.empty(int(pk.offC[-1]), dtype=torch.float64, device=DEV)
    for sa, sb, onsite, sel in _groups(pk):
        nbA, nbB, naA, naB = int(s.nbas[sa]), int(s.nbas[sb]), int(s.naux[sa]), int(s.naux[sb])
        r = torch.as_tensor(pk.dist[sel], device=DEV).reshape(-1, 1, 1, 1)
        x = torch.randn(len(sel), naA + (0 if onsite else naB), nbA, nbB, dtype=torch.float64, device=DEV,
                        generator=gen) * torch.exp(-0.8 * r)
        if onsite:
            x = torch.tril(x) + torch.tril(x, -1).transpose(2, 3)
            _put(out, pk.offC, sel, x)
        else:
            _put(out, pk.offC, sel, x)
            _put(out, pk.offC, pk.partner[sel], torch.cat([x[:, naA:], x[:, :naA]], 1).transpose(2, 3))
    return out


def _coulomb(pk, derivative=False):
    """Packed V of erfc-screened s-Gaussians, or its derivative with respect to the distance."""
    s = pk.system
    out = torch.zeros(int(pk.offV[-1]), dtype=torch.float64, device=DEV)
    for sa, sb, onsite, sel in _groups(pk):
        R = torch.as_tensor(pk.dist[sel], device=DEV).reshape(-1, 1, 1)
        p = torch.as_tensor(s.sigma[sa], device=DEV).reshape(1, -1, 1)
        q = torch.as_tensor(s.sigma[sb], device=DEV).reshape(1, 1, -1)
        g1 = torch.sqrt(2.0 * (p * p + q * q))
        g2 = torch.sqrt(g1 * g1 + 1.0 / ri.systems.OMEGA ** 2)
        Rs = torch.where(R > 0, R, torch.ones_like(R))
        v = (torch.erf(Rs / g1) - torch.erf(Rs / g2)) / Rs
        v0 = 2.0 / math.sqrt(math.pi) * (1.0 / g1 - 1.0 / g2)
        if derivative:
            e = torch.exp(-(Rs / g1) ** 2) / g1 - torch.exp(-(Rs / g2) ** 2) / g2
            v = torch.where(R > 0, 2.0 / math.sqrt(math.pi) * e / Rs - v / Rs, torch.zeros_like(v))
        else:
            v = torch.where(R > 0, v, v0)
        _put(out, pk.offV, sel, v)
        if not onsite:
            _put(out, pk.offV, pk.partner[sel], v.transpose(1, 2))
    return out


def _inputs(case, seed):
    pk = _packed(case, seed)
    gen = torch.Generator(DEV)
    gen.manual_seed(int(seed))
    x = {"pk": pk, "V": _coulomb(pk)}
    if case["task"] == "fit":
        x["eri"] = _symmetric_C(pk, gen)
        return x
    x["C"] = _symmetric_C(pk, gen)
    x["D"] = torch.as_tensor(np.concatenate([pk.gen_D(w) for w in _weights(case, pk)]), device=DEV)
    if case["task"] == "delta":
        x["K0"] = torch.randn(1 << 20, dtype=torch.float64, device=DEV, generator=gen)
    if case["task"] == "gradient":  # dC/dr = -0.8 C r/|r|, dV/dr = v'(|r|) r/|r|, per Cartesian component
        r = pk.pair_vectors()
        R = np.sqrt((r * r).sum(1))
        rhat = torch.as_tensor(np.where(R[:, None] > 0, r / np.where(R > 0, R, 1.0)[:, None], 0.0), device=DEV)
        pc = torch.repeat_interleave(rhat, torch.as_tensor(pk.sizeC, device=DEV), 0)
        pv = torch.repeat_interleave(rhat, torch.as_tensor(pk.sizeV, device=DEV), 0)
        dv = _coulomb(pk, derivative=True)
        x["dC"] = [(-0.8 * pc[:, c] * x["C"]).contiguous() for c in range(3)]
        x["dV"] = [(pv[:, c] * dv).contiguous() for c in range(3)]
    if case.get("nk"):  # points of the reciprocal cell, Gamma first
        x["k"] = np.concatenate([np.zeros((1, 3)), np.random.default_rng(seed).random((case["nk"] - 1, 3)) - 0.5])
    return x


def _old_K(K0, n):
    """The K of the iteration before (any values will do: the update is linear)."""
    return K0.repeat(-(-n // K0.numel()))[:n].contiguous()


def prepare(case, seed):
    x = _inputs(case, seed)
    s = x["pk"].system
    ex = Exchange.from_system(s, precision=case["precision"], backward=1 if case["task"] == "gradient" else 0)
    st = {"case": case, "ex": ex, **{k: v for k, v in x.items() if k != "pk"}}
    if case["task"] != "fit":
        ex.set_CV(x["C"], x["V"])
        if case["task"] != "gradient":
            st.pop("C"), st.pop("V")  # the context holds its own copy
    new = functools.partial(torch.empty, dtype=torch.float64, device=DEV)
    st["K"] = new(ex.k_elems * (2 if case["task"] == "spin" else 1))
    st["Ex"] = new(1)
    if case["task"] == "delta":
        st["K0"] = _old_K(x["K0"], ex.k_elems)
    if case.get("nk"):
        n = s.nbasis
        st["Kk"] = torch.empty(case["nk"], n, n, dtype=torch.complex128, device=DEV)
    if case["task"] == "gradient":
        st["F"] = new(3, s.n_atoms)
        st["g"] = (new(ex.d_elems), new(ex.c_elems), new(ex.v_elems))
    if case["task"] == "fit":
        st["Cfit"] = new(ex.c_elems)
    return st


# ---------------------------------------------------------------------------- one pass
def run(st):
    case, ex = st["case"], st["ex"]
    task = case["task"]
    if task == "fit":
        rix.fit_C(ex.ctx, st["V"], st["eri"], FIT_LAMBDA, st["Cfit"])
        ex.set_CV(st["Cfit"], st["V"])
        return {"C": st["Cfit"]}
    if task == "spin":
        rix.build_K_spin(ex.ctx, st["D"], st["K"], 2)
        rix.energy_spin(ex.ctx, st["D"], st["K"], st["Ex"], 2)
        return {"K": st["K"], "Ex": st["Ex"]}
    if task == "delta":
        st["K"].copy_(st["K0"])
        rix.build_K_delta(ex.ctx, st["D"], st["K"])
        return {"K": st["K"]}
    if task == "gradient":
        dD, dC, dV = ex.backward(st["D"], 1.0, *st["g"])
        for c in range(3):
            rix.force_stress(ex.ctx, c, dC, dV, st["dC"][c], st["dV"][c], st["F"][c])
        return {"dD": dD, "dC": dC, "dV": dV, "F": st["F"]}
    ex.build_K(st["D"], st["K"])
    ex.energy(st["D"], st["K"], st["Ex"])
    out = {"K": st["K"], "Ex": st["Ex"]}
    if case.get("nk"):
        rix.bloch(ex.ctx, st["K"], st["k"], st["Kk"])
        out["Kk"] = st["Kk"]
    return out


# ---------------------------------------------------------------------------- work of one pass
def _key_shift(n):
    n = np.asarray(n, np.int64)
    return (n[..., 0] << 16) + (n[..., 1] << 8) + n[..., 2]


def _kept_D(pk, w):
    """Pairs whose density block is not zero: both atoms carry an occupied orbital."""
    keep = np.zeros(pk.n_pairs, bool)
    for (atoms, img, _), wm in zip(pk.orbitals(), w):
        if wm != 0.0:
            X, Y = np.meshgrid(np.arange(len(atoms)), np.arange(len(atoms)), indexing="ij")
            k = ri.pack_key(atoms[X], atoms[Y], img[Y] - img[X]).ravel()
            pos = np.minimum(np.searchsorted(pk.keys, k), pk.n_pairs - 1)
            keep[pos[pk.keys[pos] == k]] = True
    return keep


def _reach(pk, hops):
    """Nodes reached from each atom: `hops` is a list of pair masks, one per hop."""
    rows = [np.arange(*np.searchsorted(pk.A, [a, a + 1])) for a in range(pk.system.n_atoms)]
    tail = (pk.B.astype(np.int64) << 24) + _key_shift(pk.n)  # of the pair's end, image fields unbiased
    bias = (1 << 23) + (1 << 15) + (1 << 7)
    out = []
    for a in range(pk.system.n_atoms):
        nodes = np.array([(a << 24)], np.int64)
        for keep in hops:
            new = []
            for node in nodes:
                b = (node + bias) >> 24
                p = rows[b][keep[rows[b]]]
                new.append(tail[p] + (node - (b << 24)))
            nodes = np.unique(np.concatenate(new)) if new else nodes[:0]
        out.append((nodes + bias) >> 24)
    return out


@functools.lru_cache(maxsize=64)
def _work(key):
    case = json.loads(key)
    pk = _packed(case)
    s = pk.system
    nb, na = s.nbas[s.species].astype(float), s.naux[s.species].astype(float)
    A, B, nat = pk.A, pk.B, s.n_atoms
    nC, nV, nD = int(pk.offC[-1]), int(pk.offV[-1]), int(pk.offD[-1])
    if case["task"] == "fit":  # Cholesky and two triangular solves per representative pair
        p = np.nonzero(pk.rep)[0]
        n = na[A[p]] + np.where(pk.onsite[p], 0.0, na[B[p]])
        return {"bytes": 8.0 * (nV + 2 * nC), "flops": float(np.sum(n ** 3 / 3 + 2 * n * n * nb[A[p]] * nb[B[p]]))}
    off = ~pk.onsite
    tot = lambda m: np.bincount(A, weights=m * nb[B], minlength=nat)  # noqa: E731
    sE, s1 = tot(off), tot(np.ones(len(A)))
    every = np.ones(pk.n_pairs, bool)
    n3 = [nb[x].sum() for x in _reach(pk, [every, every, every])]
    nK = float(np.sum(nb * np.array(n3)))
    flops = 0.0
    for w in _weights(case, pk):
        kD = _kept_D(pk, w)
        n2 = np.array([nb[x].sum() for x in _reach(pk, [kD, off])])
        T = np.sum(2 * na[A] * nb[A] * nb[B] * tot(kD)[B])
        U2 = np.sum(2 * na[A] * na[B] * nb[A] * nb[B])
        # term 1 once per unordered pair, term 4 once per K block
        t1 = 0.5 * np.sum(2 * na[B] * nb[A] * (na[A] + nb[B]) * s1[B])
        t2 = np.sum(2 * na * nb * s1 * sE)
        Z = np.sum(kD * 2 * na[A] * nb[B] * (na[B] + nb[A]) * sE[B])
        t4 = 0.5 * np.sum(2 * na * nb * sE * n2)
        flops += float(T + U2 + t1 + t2 + Z + t4)
    nspin = 2 if case["task"] == "spin" else 1
    byt = 8.0 * (nC + nV + nspin * (nD + nK))
    if case["task"] == "delta":
        byt += 8.0 * nK
    if case["task"] == "gradient":
        # reverse mode: each product again for either operand's adjoint; the derivative arrays once
        flops, byt = 3.0 * flops, 8.0 * (5 * (nC + nV) + 2 * nD)
    if case.get("nk"):
        byt += 16.0 * case["nk"] * s.nbasis ** 2
        flops += 4.0 * case["nk"] * nK
    return {"bytes": byt, "flops": flops}


def work(case):
    return dict(_work(json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True)))


# ---------------------------------------------------------------------------- 64-bit reference
class _Lattice:
    """Dense rows over a box of images: basis function l of atom E in cell n has column col(E, n) + l."""

    def __init__(self, pk, hops):
        s = pk.system
        self.nb = s.nbas[s.species].astype(np.int64)
        self.bo = np.concatenate([[0], np.cumsum(self.nb)])
        self.N = int(self.bo[-1])
        R = hops * np.abs(pk.n).max(axis=0).astype(np.int64)
        D = 2 * R + 1
        self.R, self.D = R, D
        self.stride = np.array([D[1] * D[2], D[2], 1]) * self.N
        self.size = int(D.prod()) * self.N
        self.origin = int((R * self.stride).sum())

    def shift(self, n):
        return int((np.asarray(n, np.int64) * self.stride).sum())

    def moved(self, cols, box):
        """The same columns in another box."""
        cell, f = cols // self.N, cols % self.N
        n = np.stack(np.unravel_index(cell, self.D), 1) - self.R
        return box.origin + n @ box.stride + f

    def cols(self, A, n):
        """Columns of the functions of several atoms A at images n, concatenated."""
        start = self.origin + (np.asarray(n, np.int64) * self.stride).sum(-1) + self.bo[A]
        cnt = self.nb[A]
        inner = np.arange(int(cnt.sum())) - np.repeat(np.cumsum(cnt) - cnt, cnt)
        return torch.as_tensor(np.repeat(start, cnt) + inner, device=DEV)


class _Reference:
    """The RI-LVL exchange contraction pair by pair (P on A; Q on the atom of k or of l)."""

    def __init__(self, pk, C, V):
        self.pk, s = pk, pk.system
        self.nat = s.n_atoms
        self.nb, self.na = s.nbas[s.species].astype(int), s.naux[s.species].astype(int)
        self.rows = [np.arange(*np.searchsorted(pk.A, [a, a + 1])) for a in range(self.nat)]
        self.g2, self.g3 = _Lattice(pk, 2), _Lattice(pk, 3)
        self.Vb = lambda p: V[pk.offV[p]:pk.offV[p + 1]].view(self.na[pk.A[p]], self.na[pk.B[p]])
        # W[A][P][i][(B, j)]: the rows of C with P on A over A's neighbours; W0 without the on-site block
        self.W, self.W0, self.nbr2, self.nbr3, self.at = [], [], [], [], {}
        for a in range(self.nat):
            blocks, blocks0, pos = [], [], 0
            for p in self.rows[a]:
                c = C[pk.offC[p]:pk.offC[p + 1]].view(-1, self.nb[a], self.nb[pk.B[p]])[:self.na[a]]
                blocks.append(c)
                blocks0.append(torch.zeros_like(c) if pk.onsite[p] else c)
                self.at[p] = pos
                pos += self.nb[pk.B[p]]
            self.W.append(torch.cat(blocks, 2))
            self.W0.append(torch.cat(blocks0, 2))
            r = self.rows[a]
            self.nbr2.append(self.g2.cols(pk.B[r], pk.n[r]))
            self.nbr3.append(self.g3.cols(pk.B[r], pk.n[r]))

    def set_D(self, D):
        pk = self.pk
        self.Db, self.Drow = {}, []
        for a in range(self.nat):
            b = [D[pk.offD[p]:pk.offD[p + 1]].view(self.nb[a], self.nb[pk.B[p]]) for p in self.rows[a]]
            self.Drow.append(torch.cat(b, 1))
            for p, d in zip(self.rows[a], b):
                self.Db[p] = d
        owner = torch.repeat_interleave(torch.arange(pk.n_pairs, device=DEV), torch.as_tensor(pk.sizeD, device=DEV))
        top = torch.zeros(pk.n_pairs, dtype=torch.float64, device=DEV).scatter_reduce(0, owner, D.abs(), "amax")
        self.has_D = (top > 0).cpu().numpy()

    def T(self, a, W=None):
        """T(A, .)[P][i][cols of the two-hop box] = sum_B C(A,B)[P on A] D(B, .)."""
        W = self.W[a] if W is None else W
        out = torch.zeros(self.na[a], self.nb[a], self.g2.size, dtype=torch.float64, device=DEV)
        for p in self.rows[a]:
            b = self.pk.B[p]
            x = W[:, :, self.at[p]:self.at[p] + self.nb[b]] @ self.Drow[b]
            out.index_add_(2, self.nbr2[b] + self.g2.shift(self.pk.n[p]), x)
        return out

    def node2(self, p):
        c = self.g2.origin + self.g2.shift(self.pk.n[p]) + int(self.g2.bo[self.pk.B[p]])
        return slice(c, c + self.nb[self.pk.B[p]])

    def node3(self, p):
        c = self.g3.origin + self.g3.shift(self.pk.n[p]) + int(self.g3.bo[self.pk.B[p]])
        return slice(c, c + self.nb[self.pk.B[p]])

    def Z(self, b, scale):
        """scale * sum_G D(B,G) V(B,G) C(G, .)[Q on G], the on-site C block left out."""
        out = torch.zeros(self.na[b], self.nb[b], self.g2.size, dtype=torch.float64, device=DEV)
        for p in self.rows[b]:
            if self.has_D[p]:
                g = self.pk.B[p]
                W = self.W0[g]
                F = (self.Vb(p) @ W.reshape(self.na[g], -1)).view(self.na[b], self.nb[g], -1)
                out.index_add_(2, self.nbr2[g] + self.g2.shift(self.pk.n[p]), scale * (self.Db[p] @ F))
        return out

    def X(self):
        """Rows of terms 1, 2 and 4 (half of 1 and 4), so that K = X + X^T with term 3 the transpose of 2."""
        pk = self.pk
        X = torch.zeros(self.g3.N, self.g3.size, dtype=torch.float64, device=DEV)
        for a in range(self.nat):
            Xa = X[int(self.g3.bo[a]):int(self.g3.bo[a + 1])]
            T = self.T(a)
            for p in self.rows[a]:
                e = pk.B[p]
                V = self.Vb(p)
                sh = pk.n[p]
                # term 1: P on A, Q on E
                t = T.index_select(2, self.nbr2[e] + self.g2.shift(sh))
                U = (V.T @ t.reshape(self.na[a], -1)).view(self.na[e], self.nb[a], -1)
                w = self.W[e].permute(0, 2, 1).reshape(-1, self.nb[e])
                Xa[:, self.node3(p)] += 0.5 * (U.transpose(0, 1).reshape(self.nb[a], -1) @ w)
                # term 2: P on A, Q on G
                U = (V.T @ T[:, :, self.node2(p)].reshape(self.na[a], -1)).view(self.na[e], self.nb[a], -1)
                x = U.transpose(0, 1).reshape(self.nb[a], -1) @ self.W0[e].reshape(-1, self.W0[e].shape[2])
                Xa.index_add_(1, self.nbr3[e] + self.g3.shift(sh), x)
        for b in range(self.nat):
            Z = self.Z(b, 0.5)
            used = torch.nonzero((Z != 0).any(0).any(0)).reshape(-1)
            Zc = Z.index_select(2, used).reshape(self.na[b] * self.nb[b], -1)
            del Z
            c3 = torch.as_tensor(self.g2.moved(used.cpu().numpy(), self.g3), device=DEV)
            for p in self.rows[b]:  # pair (A, B, -n) of the pair (B, A, n)
                if pk.onsite[p]:
                    continue
                a = pk.B[p]
                w = self.W[b][:, :, self.at[p]:self.at[p] + self.nb[a]].reshape(-1, self.nb[a])
                X[int(self.g3.bo[a]):int(self.g3.bo[a + 1])].index_add_(1, c3 - self.g3.shift(pk.n[p]), w.T @ Zc)
        return X

    def k_pattern(self):
        """(A, E, n) of the K blocks, sorted: every node three pair hops from A."""
        pk = self.pk
        bias = (1 << 23) + (1 << 15) + (1 << 7)
        tail = (pk.B.astype(np.int64) << 24) + _key_shift(pk.n)
        keys = []
        for a in range(self.nat):
            nodes = np.array([a << 24], np.int64)
            for _ in range(3):
                nodes = np.unique(np.concatenate(
                    [tail[self.rows[(x + bias) >> 24]] + (x - (((x + bias) >> 24) << 24)) for x in nodes]))
            keys.append((np.int64(a) << 44) + nodes + bias)
        return ri.unpack_key(np.concatenate(keys))

    def pack_K(self, X):
        A, E, n = self.k_pattern()
        nb = self.nb.astype(np.int64)
        off = np.concatenate([[0], np.cumsum(nb[A] * nb[E])])
        K = torch.empty(int(off[-1]), dtype=torch.float64, device=DEV)
        sp = self.pk.system.species
        code = sp[A].astype(np.int64) * 64 + sp[E]
        ca = self.g3.origin + n.astype(np.int64) @ self.g3.stride
        cb = self.g3.origin - n.astype(np.int64) @ self.g3.stride
        flat = X.reshape(-1)
        for g in np.unique(code):
            sel = np.nonzero(code == g)[0]
            for part in np.array_split(sel, -(-len(sel) // 200000)):
                a, e = A[part], E[part]
                i = torch.arange(int(nb[a[0]]), device=DEV).reshape(1, -1, 1)
                el = torch.arange(int(nb[e[0]]), device=DEV).reshape(1, 1, -1)
                dev = lambda v: torch.as_tensor(v, device=DEV).reshape(-1, 1, 1)  # noqa: E731
                bo = self.g3.bo
                x = flat[(dev(bo[a]) + i) * self.g3.size + dev(ca[part] + bo[e]) + el]
                x = x + flat[(dev(bo[e]) + el) * self.g3.size + dev(cb[part] + bo[a]) + i]
                _put(K, off, part, x)
        return K, (A, E, n, off)

    def energy(self, X, scale=-0.25):
        """scale * sum over pairs <D(E,A,-n), K(A,E,n)>, with K = X + X^T."""
        e = torch.zeros((), dtype=torch.float64, device=DEV)
        for a in range(self.nat):
            Xa = X[int(self.g3.bo[a]):int(self.g3.bo[a + 1])]
            e += (self.Drow[a] * Xa.index_select(1, self.nbr3[a])).sum()
        return (2.0 * scale * e).reshape(1)

    def bloch(self, K, pattern, kfrac):
        A, E, n, off = pattern
        N = self.g3.N
        out = torch.zeros(len(kfrac), N * N, dtype=torch.complex128, device=DEV)
        sp, nb, bo = self.pk.system.species, self.nb.astype(np.int64), self.g3.bo
        code = sp[A].astype(np.int64) * 64 + sp[E]
        for g in np.unique(code):
            for part in np.array_split(np.nonzero(code == g)[0], -(-int((code == g).sum()) // 200000)):
                i = torch.arange(int(nb[A[part[0]]]), device=DEV).reshape(1, -1, 1)
                el = torch.arange(int(nb[E[part[0]]]), device=DEV).reshape(1, 1, -1)
                dev = lambda v: torch.as_tensor(v, device=DEV).reshape(-1, 1, 1)  # noqa: E731
                x = K[dev(off[part]) + i * int(nb[E[part[0]]]) + el]
                at = ((dev(bo[A[part]]) + i) * N + dev(bo[E[part]]) + el).reshape(-1)
                for q, k in enumerate(np.asarray(kfrac)):
                    ph = torch.as_tensor(2.0 * math.pi * (n[part] @ k), device=DEV).reshape(-1, 1, 1)
                    z = torch.complex(x * torch.cos(ph), x * torch.sin(ph))
                    out[q].index_add_(0, at, z.reshape(-1))
        return out.view(len(kfrac), N, N)

    def gradients(self):
        """dE/dC^P = -1/2 D M^P D with M^P = sum_Q V_PQ C^Q, and dE/dV_PQ = -1/4 Tr(D C^P D C^Q)."""
        pk = self.pk
        dC = torch.zeros(int(pk.offC[-1]), dtype=torch.float64, device=DEV)
        dV = torch.zeros(int(pk.offV[-1]), dtype=torch.float64, device=DEV)
        T = [self.T(a) for a in range(self.nat)]
        T0 = [self.T(a, self.W0[a]) for a in range(self.nat)]
        for a in range(self.nat):
            # L^P = D_A M^P: Q on G, the rows of C^Q from G (with its on-site block) and the columns at G
            L = self.Z(a, 1.0)
            for p in self.rows[a]:
                g, q = pk.B[p], pk.partner[p]
                back = self.node2(q)  # A seen from G
                L[:, :, self.node2(p)] += torch.einsum("pq,qki->pik", self.Vb(p), T[g][:, :, back])
                # dV(A,G): W~ = 2 W0 + on-site block
                t = T[g][:, :, back] + T0[g][:, :, back]
                g1 = torch.einsum("qka,pak->pq", t, T[a][:, :, self.node2(p)])
                w = torch.einsum("ak,qkx->qax", self.Db[p], self.W[g] + self.W0[g]).reshape(self.na[g], -1)
                t0 = T0[a].index_select(2, self.nbr2[g] + self.g2.shift(pk.n[p])).reshape(self.na[a], -1)
                dV[pk.offV[p]:pk.offV[p + 1]] = -0.25 * (g1 + t0 @ w.T).reshape(-1)
            for p in self.rows[a]:
                b, q = pk.B[p], pk.partner[p]
                l = L.index_select(2, self.nbr2[b] + self.g2.shift(pk.n[p]))
                own = -0.5 * torch.einsum("pix,jx->pij", l, self.Drow[b])
                if pk.onsite[p]:
                    own = 0.5 * (own + own.transpose(1, 2))
                    dC[pk.offC[p]:pk.offC[p + 1]] = own.reshape(-1)
                else:
                    n = own.numel()
                    dC[pk.offC[p]:pk.offC[p] + n] = own.reshape(-1)
                    dC[pk.offC[q + 1] - n:pk.offC[q + 1]] = own.transpose(1, 2).reshape(-1)
        return dC, dV


def _exact_fit(x):
    pk = x["pk"]
    s = pk.system
    out = torch.empty_like(x["eri"])
    onsite = np.full(s.n_atoms, -1)
    onsite[pk.A[pk.onsite]] = np.nonzero(pk.onsite)[0]

    def blocks(arr, off, sel, shape):
        start = torch.as_tensor(off[sel], device=DEV)
        return arr[start[:, None] + torch.arange(int(np.prod(shape)), device=DEV)].view(len(sel), *shape)

    for sa, sb, ons, sel in _groups(pk):
        na, nb = int(s.naux[sa]), int(s.naux[sb])
        M = blocks(x["V"], pk.offV, onsite[pk.A[sel]], (na, na))
        if not ons:
            ab = blocks(x["V"], pk.offV, sel, (na, nb))
            bb = blocks(x["V"], pk.offV, onsite[pk.B[sel]], (nb, nb))
            M = torch.cat([torch.cat([M, ab], 2), torch.cat([ab.transpose(1, 2), bb], 2)], 1)
        M = M + FIT_LAMBDA * torch.eye(M.shape[1], dtype=M.dtype, device=DEV)
        fa, fb = int(s.nbas[sa]), int(s.nbas[sb])
        e = blocks(x["eri"], pk.offC, sel, (M.shape[1], fa * fb))
        c = torch.cholesky_solve(e, torch.linalg.cholesky(M)).view(len(sel), -1, fa, fb)
        _put(out, pk.offC, sel, c)
        if not ons:
            _put(out, pk.offC, pk.partner[sel], torch.cat([c[:, na:], c[:, :na]], 1).transpose(2, 3))
    return {"C": out}


def exact(case, seed):
    x = _inputs(case, seed)
    pk = x["pk"]
    if case["task"] == "fit":
        return _exact_fit(x)
    if case["system"] == "ice" and case["nx"] * case["ny"] * case["nz"] > 4:
        return None  # over half a minute
    ref = _Reference(pk, x["C"], x["V"])
    nD = int(pk.offD[-1])
    K, E = [], []
    for c in range(x["D"].numel() // nD):
        ref.set_D(x["D"][c * nD:(c + 1) * nD].contiguous())
        X = ref.X()
        k, pattern = ref.pack_K(X)
        K.append(k)
        E.append(ref.energy(X, -0.5 if case["task"] == "spin" else -0.25))
        del X
    if case["task"] == "delta":
        return {"K": _old_K(x["K0"], K[0].numel()) + K[0]}
    if case["task"] == "gradient":
        dC, dV = ref.gradients()
        A, E_, n, off = pattern
        at = {int(k): i for i, k in enumerate(ri.pack_key(A, E_, n))}
        dD = torch.cat([-0.5 * K[0][off[at[int(k)]]:off[at[int(k)] + 1]] for k in pk.keys])
        F = torch.zeros(3, pk.system.n_atoms, dtype=torch.float64, device=DEV)
        pC = torch.repeat_interleave(torch.arange(pk.n_pairs, device=DEV), torch.as_tensor(pk.sizeC, device=DEV))
        pV = torch.repeat_interleave(torch.arange(pk.n_pairs, device=DEV), torch.as_tensor(pk.sizeV, device=DEV))
        first = torch.as_tensor(pk.A.astype(np.int64), device=DEV)
        partner = torch.as_tensor(pk.partner, device=DEV)
        for c in range(3):
            g = torch.zeros(pk.n_pairs, dtype=torch.float64, device=DEV)
            g.index_add_(0, pC, dC * x["dC"][c]).index_add_(0, pV, dV * x["dV"][c])
            F[c].index_add_(0, first, g - g[partner])
        return {"dD": dD, "dC": dC, "dV": dV, "F": F}
    out = {"K": torch.cat(K), "Ex": sum(E)}
    if case.get("nk"):
        out["Kk"] = ref.bloch(K[0], pattern, x["k"])
    return out
