"""What a user of this framework has it do, as cases with inputs, one pass and an independent 64-bit answer.

A pass goes through the public entry points of ``paper_2310_05279_gb300`` only: ``D3.compute``,
``D3.compute_batch``, ``D3.compute_batch_host``, ``D3Function`` with its backward, and
``heat_current``.  The systems come from the package's own generators:

    sheet    one AB-stacked graphene bilayer of nx x ny rectangles (8 nx ny C atoms)
    scan     n_dist x n_slide such bilayers, the binding and sliding scan
    box      one periodic H/C/N/O/Zn box of 4 ncell^3 atoms at 1.0 g/cm^3
    uneven   a batch of triclinic H/C/N/O/Cu/Zn structures with log-uniform sizes

and the kinds of pass are:

    call     one structure per call (a relaxation or a short MD run without list reuse)
    batch    a whole batch per call; optionally with site energies and coordination numbers
    md       a molecular-dynamics step with list reuse: positions move, the list is kept by the skin
    heat     the step of a thermal-conductivity run: per-atom virials, then the heat current
    npt      a step of a run whose cell changes: every call brings a new cell
    dataset  structures streamed from host arrays, another batch in every call
    refit    a step of a damping refit: energies, forces, loss and its gradients

The precision ("mixed" or "fp64") is the handle's option; ``s9`` turns on the three-body term.
"""
import math

import numpy as np
import torch

import paper_2310_05279_gb300 as d3gb
from paper_2310_05279_gb300 import D3, heat_current, workloads as wl

BOHR = 0.529177210903
HARTREE = 27.211386245988


def listed():
    return [
        # the smallest call: one 64-atom cell, as an MD or relaxation loop around a short-range model makes it
        dict(name="single_64", kind="call", system="sheet", nx=2, ny=4, precision="mixed"),
        # the binding/sliding scan, 128 bilayers of 1,440 atoms in one call: the headline workload
        dict(name="scan", kind="batch", system="scan", n_dist=16, n_slide=8, nx=10, ny=18, precision="mixed"),
        # the same in the plain FP64 form, which checks and reference data are made with
        dict(name="scan_fp64", kind="batch", system="scan", n_dist=16, n_slide=8, nx=10, ny=18, precision="fp64"),
        # one box of 1,048,576 atoms of five elements: the largest call
        dict(name="box_1m", kind="batch", system="box", ncell=64, precision="mixed"),
        # 512 structures of 50 to 4000 atoms, with site energies and coordination numbers: screening a data set
        dict(name="uneven_512", kind="batch", system="uneven", nstruct=512, lo=50, hi=4000, precision="mixed",
             atoms=True),
        # a step of molecular dynamics of a 131,072-atom box with a 0.5 A skin
        dict(name="md_box", kind="md", system="box", ncell=32, precision="mixed", skin=0.5),
        # a thermal-conductivity step of a 55,296-atom box of MOF composition: per-atom virials and heat current
        dict(name="heat_box", kind="heat", system="box", ncell=24, precision="mixed"),
        # a step at changing cell (NPT or cell relaxation) of a 6,912-atom box
        dict(name="npt_box", kind="npt", system="box", ncell=12, precision="mixed"),
        # structures streamed from host arrays, 64 at a time, every call another batch
        dict(name="dataset_host", kind="dataset", system="uneven", nstruct=64, lo=50, hi=4000, precision="mixed"),
        # the scan with the optional three-body term
        dict(name="scan_atm", kind="batch", system="scan", n_dist=16, n_slide=8, nx=10, ny=18, precision="mixed",
             s9=1.0),
        # a step of a damping refit over 256 structures of 200 to 2000 atoms
        dict(name="refit", kind="refit", system="uneven", nstruct=256, lo=200, hi=2000, precision="mixed"),
        # the same in FP64 on a smaller batch, as a refit is checked or finished
        dict(name="refit_fp64", kind="refit", system="uneven", nstruct=32, lo=200, hi=2000, precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["call", "batch", "batch", "batch", "md", "heat", "npt", "dataset", "refit"])
    fp64 = rng.random() < 0.3
    c = dict(kind=kind, precision="fp64" if fp64 else "mixed")
    if kind == "call":
        if rng.random() < 0.5:
            c.update(system="sheet", nx=rng.randint(2, 12), ny=rng.randint(3, 20))
        else:
            c.update(system="box", ncell=rng.randint(3, 10))
    elif kind == "batch":
        system = rng.choice(["scan", "box", "uneven"])
        c["system"] = system
        if system == "scan":
            c.update(n_dist=rng.randint(2, 16), n_slide=rng.randint(1, 8), nx=rng.randint(3, 10), ny=rng.randint(5, 18))
            if rng.random() < 0.3:
                c["s9"] = 1.0
        elif system == "box":
            c.update(ncell=rng.randint(6, 28 if fp64 else 63))
        else:
            c.update(nstruct=_log_int(rng, 4, 100 if fp64 else 500), lo=rng.randint(20, 200), hi=rng.randint(400, 4000),
                     atoms=rng.random() < 0.5)
    elif kind == "md":
        c.update(system="box", ncell=rng.randint(6, 20 if fp64 else 36), skin=rng.choice([0.5, 0.75, 1.0]))
    elif kind == "heat":
        c.update(system="box", ncell=rng.randint(5, 18 if fp64 else 30))
    elif kind == "npt":
        c.update(system="box", ncell=rng.randint(4, 24))
    elif kind == "dataset":
        c.update(system="uneven", nstruct=_log_int(rng, 4, 64), lo=rng.randint(20, 200), hi=rng.randint(400, 4000))
    else:
        c.update(system="uneven", nstruct=_log_int(rng, 4, 32 if fp64 else 256), lo=rng.randint(50, 300),
                 hi=rng.randint(500, 2000))
    return c


# ------------------------------------------------------------------ inputs

def _batch(case, seed):
    system = case["system"]
    if system == "sheet":
        g = np.random.Generator(np.random.PCG64(seed))
        s = wl.bilayer(case["nx"], case["ny"], 3.4, wl.BOND, 20.0, 0.02, g)
        return wl.batch_of([s], wl.carbon_table(1000))
    if system == "scan":
        return wl.bilayer_scan(seed=seed, n_dist=case["n_dist"], n_slide=case["n_slide"], nx=case["nx"], ny=case["ny"])
    if system == "box":
        return wl.mof_like_box(seed=seed, ncell=case["ncell"])
    # sizes (log-uniform, of the case), then the structures as wl.uneven_batch draws them
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    sizes = np.exp(np.random.Generator(np.random.PCG64(case["nstruct"])).uniform(lo, hi, case["nstruct"]))
    g = np.random.Generator(np.random.PCG64(seed))
    structs = [wl.random_structure(g, int(round(n)), wl.UNEVEN_ELEMENTS) for n in sizes]
    return wl.batch_of(structs, wl.random_tables(wl.UNEVEN_ELEMENTS, 1003))


def _params(case):
    p = dict(wl.PBE_BJ)
    if case.get("s9"):
        p.update(s9=case["s9"], alpha9=16.0, rc3=6.0)
    return p


_STRAIN = (0.0, 0.0020, -0.0013, 0.0008)  # of the cells that an "npt" state's calls go through
_MD_STEPS = 16                            # displacements of an "md" state's calls: a triangular wave


def _md_amplitude(k, skin):
    """Displacement scale of step k: 0.15 skin a step, so that the list is rebuilt every fourth step or so."""
    k %= _MD_STEPS
    up = min(k, 8 - k) if k <= 8 else -min(k - 8, 16 - k)
    return 0.15 * skin * up


def _md_direction(n, seed):
    """A displacement of at most 1 A per atom."""
    g = np.random.Generator(np.random.PCG64(seed + 77))
    v = g.normal(size=(n, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True) * g.uniform(0.2, 1.0, (n, 1))


def _targets(b, seed):
    """Reference energies and forces of a refit."""
    g = np.random.Generator(np.random.PCG64(seed + 55))
    n = np.diff(b.offsets).astype(np.float64)
    return -n * g.uniform(0.02, 0.3, len(n)), 0.05 * g.normal(size=(b.natoms, 3))


def prepare(case, seed):
    kind = case["kind"]
    b = _batch(case, seed)
    d3 = D3(b.tables, _params(case), precision=case["precision"], skin=case.get("skin", 0.0))
    st = dict(kind=kind, case=case, d3=d3, b=b, k=0)
    if kind == "dataset":
        other = _batch(case, seed + 1_000_003)
        st["batches"] = [b, other]
        return st
    st["pos"] = torch.tensor(b.pos, dtype=torch.float64, device="cuda")
    st["typ"] = torch.tensor(b.types, dtype=torch.int32, device="cuda")
    if kind == "md":
        st["pos0"] = st["pos"].clone()
        st["dir"] = torch.tensor(_md_direction(b.natoms, seed), device="cuda")
        st["out"] = dict(E=torch.empty(b.nstruct, dtype=torch.float64, device="cuda"),
                         F=torch.empty((b.natoms, 3), dtype=torch.float64, device="cuda"),
                         W=torch.empty((b.nstruct, 3, 3), dtype=torch.float64, device="cuda"))
    elif kind == "heat":
        st["vel"] = torch.tensor(wl.maxwell_velocities(wl.atom_masses(b), 300.0, seed), device="cuda")
    elif kind == "npt":
        st["cells"] = [b.cells[0] * (1.0 + e) for e in _STRAIN]
        st["poses"] = [st["pos"] * (1.0 + e) for e in _STRAIN]
    elif kind == "refit":
        e, f = _targets(b, seed)
        st["pos"].requires_grad_(True)
        st["theta"] = torch.tensor([wl.PBE_BJ[k] for k in ("s6", "s8", "a1", "a2")], dtype=torch.float64,
                                   device="cuda", requires_grad=True)
        st["Eref"] = torch.tensor(e, device="cuda")
        st["Fref"] = torch.tensor(f, device="cuda")
        st["n"] = torch.tensor(np.diff(b.offsets).astype(np.float64), device="cuda")
    return st


def _loss(E, F, Eref, Fref, n):
    return (((E - Eref) / n) ** 2).mean() + 0.1 * ((F - Fref) ** 2).mean()


def run(st):
    kind, d3, b = st["kind"], st["d3"], st["b"]
    if kind == "call":
        return d3.compute(st["pos"], st["typ"], b.cells[0], b.pbc[0])
    if kind == "batch":
        atoms = bool(st["case"].get("atoms"))
        return d3.compute_batch(st["pos"], st["typ"], b.offsets, b.cells, b.pbc, e_atom=atoms, cn=atoms)
    if kind == "md":
        torch.add(st["pos0"], st["dir"], alpha=_md_amplitude(st["k"], st["case"]["skin"]), out=st["pos"])
        st["k"] += 1
        return d3.compute_batch(st["pos"], st["typ"], b.offsets, b.cells, b.pbc, out=st["out"])
    if kind == "heat":
        out = d3.compute_batch(st["pos"], st["typ"], b.offsets, b.cells, b.pbc, w_atom=True)
        out["J"] = heat_current(out["w_atom"], st["vel"])
        return out
    if kind == "npt":
        k = st["k"] % len(_STRAIN)
        st["k"] += 1
        return d3.compute(st["poses"][k], st["typ"], st["cells"][k], b.pbc[0])
    if kind == "dataset":
        x = st["batches"][st["k"] % 2]
        st["k"] += 1
        return d3.compute_batch_host(x.pos, x.types, x.offsets, x.cells, x.pbc)
    st["pos"].grad = st["theta"].grad = None
    E, F = d3gb.D3Function.apply(st["pos"], st["theta"], d3, st["typ"], b.offsets, b.cells, b.pbc)
    _loss(E, F, st["Eref"], st["Fref"], st["n"]).backward()
    return dict(E=E.detach(), F=F.detach(), dpos=st["pos"].grad, dtheta=st["theta"].grad)


# ------------------------------------------------------------------ work

# pairs within 12 A and within 6 A per atom (each pair once): counted on the bilayer and on the box; for the uneven
# structures the expectation over their densities and element mixes
_PAIRS = {"sheet": (152.0, 25.0), "scan": (152.0, 25.0), "box": (210.0, 26.0), "uneven": (132.0, 16.5)}
_NREF = {"sheet": 5.0, "scan": 5.0, "box": 3.2, "uneven": 2.2}


def _atoms(case):
    s = case["system"]
    if s == "sheet":
        return 8 * case["nx"] * case["ny"], 1
    if s == "scan":
        return case["n_dist"] * case["n_slide"] * 8 * case["nx"] * case["ny"], case["n_dist"] * case["n_slide"]
    if s == "box":
        return 4 * case["ncell"] ** 3, 1
    lo, hi = case["lo"], case["hi"]
    return case["nstruct"] * (hi - lo) / math.log(hi / lo), case["nstruct"]


def work(case):
    """Positions and types read, results written; each pair of Eq. 2 once (53 + 6 Nref operations: distance, the C6
    interpolation with both derivatives, damping, energy, forces and virial) and each pair of Eq. 4 once (about 60)."""
    n, b = _atoms(case)
    pd, pc = _PAIRS[case["system"]]
    nref = _NREF[case["system"]]
    flops = n * (pd * (53 + 6 * nref) + pc * 60)
    nbytes = n * (24 + 4 + 24) + b * (72 + 8 + 72 + 12)
    if case.get("atoms"):
        nbytes += 16 * n
    if case.get("s9"):
        flops += n * 244.0 * (183 + 2 * nref)  # 244 triangles per atom below 6 A on the bilayer
    if case["kind"] == "heat":
        flops += n * (2 * pc * 45 + 15)
        nbytes += n * (72 + 24 + 24)
    if case["kind"] == "refit":
        flops *= 3  # a derivative along one direction of every force term costs about two evaluations more
        nbytes += n * (24 + 24) + 64
    return {"bytes": float(nbytes), "flops": float(flops)}


# ------------------------------------------------------------------ the same in 64 bits, plain torch

class _System:
    """A batch in bohr on the GPU with its periodic images, binned for the pair search."""

    def __init__(self, pos, types, offsets, cells, pbc, rc):
        dev = "cuda"
        n = len(pos)
        nst = len(offsets) - 1
        sid = np.repeat(np.arange(nst), np.diff(offsets))
        H = torch.tensor(np.asarray(cells).reshape(-1, 3, 3) / BOHR, device=dev)
        self.sid = torch.tensor(sid, device=dev)
        self.nst, self.n, self.rc = nst, n, rc
        self.typ = torch.tensor(np.asarray(types), dtype=torch.int64, device=dev)
        x = torch.tensor(np.asarray(pos) / BOHR, device=dev)
        per = torch.tensor(np.asarray(pbc).reshape(-1, 3), device=dev).bool()
        Ha, pa = H[self.sid], per[self.sid]
        f = torch.linalg.solve(Ha.transpose(1, 2), x.unsqueeze(-1)).squeeze(-1)
        f = torch.where(pa, f - torch.floor(f), f)
        self.x = (f.unsqueeze(1) @ Ha).squeeze(1)
        vol = torch.linalg.det(H).abs()
        cr = torch.stack([torch.linalg.cross(H[:, (k + 1) % 3], H[:, (k + 2) % 3]) for k in range(3)], 1)
        delta = rc * cr.norm(dim=2) / vol[:, None] + 1e-9
        m = torch.where(per, torch.ceil(delta), torch.zeros_like(delta)).amax(0).long().tolist() if nst else [0, 0, 0]
        da = torch.where(pa, delta[self.sid], torch.full_like(delta[self.sid], 1e9))
        src, sh = [], []
        for a in range(-m[0], m[0] + 1):
            for b in range(-m[1], m[1] + 1):
                for c in range(-m[2], m[2] + 1):
                    t = torch.tensor([a, b, c], dtype=torch.float64, device=dev)
                    g = f + t
                    ok = ((g >= -da) & (g < 1 + da) & (pa | (t == 0))).all(1)
                    k = ok.nonzero().squeeze(1)
                    src.append(k)
                    sh.append((t.expand(len(k), 3).unsqueeze(1) @ Ha[k]).squeeze(1))
        self.src, self.sh = torch.cat(src), torch.cat(sh)
        y = self.x[self.src] + self.sh
        ys = self.sid[self.src]
        lo = torch.full((nst, 3), 1e30, dtype=torch.float64, device=dev).scatter_reduce(
            0, ys[:, None].expand(-1, 3), y, "amin")
        hi = torch.full((nst, 3), -1e30, dtype=torch.float64, device=dev).scatter_reduce(
            0, ys[:, None].expand(-1, 3), y, "amax")
        nb = ((hi - lo) / rc).floor().clamp(min=0).long() + 3  # one empty bin on each side
        self.nb, self.lo = nb, lo
        tot = nb.prod(1)
        self.base = torch.cumsum(tot, 0) - tot
        order = torch.argsort(self._key(y, ys), stable=True)
        self.src, self.sh = self.src[order], self.sh[order]
        self.keys = self._key(y[order], ys[order])

    def _bins(self, y, s):
        return ((y - self.lo[s]) / self.rc).floor().long() + 1

    def _key(self, y, s):
        b, nb = self._bins(y, s), self.nb[s]
        return self.base[s] + (b[:, 2] * nb[:, 1] + b[:, 1]) * nb[:, 0] + b[:, 0]

    def pairs(self, rc, per_chunk):
        """Chunks (i, j, shift) of ordered pairs with |x_j + shift - x_i| < rc <= self.rc."""
        for a in range(0, self.n, per_chunk):
            i = torch.arange(a, min(self.n, a + per_chunk), device="cuda")
            s = self.sid[i]
            b, nb = self._bins(self.x[i], s), self.nb[s]
            los, his = [], []
            for dz in (-1, 0, 1):
                for dy in (-1, 0, 1):
                    k = self.base[s] + ((b[:, 2] + dz) * nb[:, 1] + b[:, 1] + dy) * nb[:, 0] + b[:, 0]
                    los.append(torch.searchsorted(self.keys, k - 1))
                    his.append(torch.searchsorted(self.keys, k + 1, right=True))
            lo, cnt = torch.stack(los, 1).reshape(-1), (torch.stack(his, 1) - torch.stack(los, 1)).reshape(-1)
            ii = i.repeat_interleave(9).repeat_interleave(cnt)
            first = (torch.cumsum(cnt, 0) - cnt).repeat_interleave(cnt)
            e = lo.repeat_interleave(cnt) + torch.arange(len(ii), device="cuda") - first
            j, sh = self.src[e], self.sh[e]
            d2 = ((self.x[j] + sh - self.x[ii]) ** 2).sum(1)
            k = ((d2 < rc * rc) & ~((j == ii) & (sh == 0).all(1))).nonzero().squeeze(1)
            yield ii[k], j[k], sh[k]


def _add(n, i, v):
    return torch.zeros((n,) + v.shape[1:], dtype=torch.float64, device="cuda").index_add(0, i, v)


def _d3_64(S, tab, prm, x, theta, site=False, parts=False):
    """Eqs. 1-7 in 64 bits.  x (n, 3) bohr and theta = (s6, s8, a1, a2) may carry forward-mode tangents."""
    dev = "cuda"
    s6, s8, a1, a2 = theta[0], theta[1], theta[2], theta[3]
    k1, k2, k3 = prm["k1"], prm["k2"], prm["k3"]
    n, t = S.n, S.typ
    rk = k2 * torch.tensor(tab.rcov, device=dev)
    sq = torch.tensor(tab.sqrtq, device=dev)
    nref = torch.tensor(tab.nref, device=dev)
    R = int(tab.max_ref)
    cnr = torch.tensor(tab.cn_ref, device=dev)
    c6r = torch.tensor(tab.c6_ref, device=dev)  # [ti, tj, a, b]
    valid = torch.arange(R, device=dev)[None, :] < nref[:, None]
    c6r = c6r * valid[:, None, :, None] * valid[None, :, None, :]
    rcn = prm["rc_cn"] / BOHR
    cn = torch.zeros(n, dtype=torch.float64, device=dev)
    near = list(S.pairs(rcn, 16384))
    for i, j, sh in near:
        r = (x[j] + sh - x[i]).pow(2).sum(1).sqrt()
        cn = cn + _add(n, i, 1.0 / (1.0 + torch.exp(-k1 * ((rk[t[i]] + rk[t[j]]) / r - 1.0))))
    z = cn[:, None] - cnr[t]
    ex = torch.where(valid[t], -k3 * z * z, torch.full_like(z, -1e300))
    W = torch.exp(ex - ex.detach().amax(1, keepdim=True)) * valid[t]
    W = W / W.sum(1, keepdim=True)
    dW = W * (-2 * k3 * z + (W * 2 * k3 * z).sum(1, keepdim=True))
    v = torch.stack([torch.einsum("nab,nb->na", c6r[u][t], W) for u in range(len(tab.nref))], 1)  # [n, type, a]
    U = torch.zeros(n, dtype=torch.float64, device=dev)
    dEdn, F = torch.zeros_like(U), torch.zeros((n, 3), dtype=torch.float64, device=dev)
    D = torch.zeros((n if parts else S.nst, 3, 3), dtype=torch.float64, device=dev)
    P = torch.zeros((n, 3), dtype=torch.float64, device=dev)
    home = (lambda i: i) if parts else (lambda i: S.sid[i])
    for i, j, sh in S.pairs(prm["rc_disp"] / BOHR, 8192):
        d = x[j] + sh - x[i]
        r2 = d.pow(2).sum(1)
        q = 3.0 * sq[t[i]] * sq[t[j]]
        rad = a1 * q.sqrt() + a2
        vj = v[j, t[i]]
        C6, dC6 = (W[i] * vj).sum(1), (dW[i] * vj).sum(1)
        d6, d8 = r2 ** 3 + rad ** 6, r2 ** 4 + rad ** 8
        g = s6 / d6 + s8 * q / d8
        U = U + _add(n, i, -0.5 * C6 * g)
        dEdn = dEdn + _add(n, i, -g * dC6)
        fd = (C6 * (6 * r2 ** 2 * s6 / d6 ** 2 + 8 * r2 ** 3 * s8 * q / d8 ** 2))[:, None] * d
        F = F + _add(n, i, fd)
        D = D + _add(len(D), home(i), -0.5 * fd[:, :, None] * d[:, None, :])
        if parts:
            P = P + _add(n, i, (-0.5 * g * dC6)[:, None] * d)
    if prm.get("s9"):
        e3, f3, w3, gn = _three_body(S, tab, prm, x, W, dW, c6r, theta)
        U, F, dEdn, D = U + e3, F + f3, dEdn + gn, D + w3
    out = dict(U=U, cn=cn)
    G, M = torch.zeros((n, 3), dtype=torch.float64, device=dev), 0.0
    for i, j, sh in near:
        d = x[j] + sh - x[i]
        r = d.pow(2).sum(1).sqrt()
        rc = rk[t[i]] + rk[t[j]]
        f = 1.0 / (1.0 + torch.exp(-k1 * (rc / r - 1.0)))
        c = -k1 * rc * f * (1.0 - f) / r ** 3  # f'(r) / r
        F = F + _add(n, i, ((dEdn[i] + dEdn[j]) * c)[:, None] * d)
        if parts:
            dd = d[:, :, None] * d[:, None, :]
            D = D + _add(n, i, -(dEdn[j] * c)[:, None, None] * dd)
            M = M + _add(n, i, c[:, None, None] * P[j][:, :, None] * d[:, None, :])
            G = G + _add(n, i, c[:, None] * d)
        else:
            D = D + _add(len(D), home(i), -(dEdn[i] * c)[:, None, None] * d[:, :, None] * d[:, None, :])
    E = torch.zeros(S.nst, dtype=torch.float64, device=dev).index_add(0, S.sid, U)
    out.update(E=E * HARTREE, F=F * (HARTREE / BOHR))
    if parts:
        wa = (D - P[:, :, None] * G[:, None, :] - M) * HARTREE
        out["w_atom"] = wa
        out["W"] = torch.zeros((S.nst, 3, 3), dtype=torch.float64, device=dev).index_add(0, S.sid, wa)
    else:
        out["W"] = D * HARTREE
    if site:
        out["e_atom"] = U * HARTREE
    return out


def _three_body(S, tab, prm, x, W, dW, c6r, theta):
    """The triple-dipole term from every vertex of every triangle: site energies, forces, virial, dE/dn."""
    t, n = S.typ, S.n
    sq = torch.tensor(tab.sqrtq, device="cuda")
    rc3, third = prm["rc3"] / BOHR, prm["alpha9"] / 3.0
    U = torch.zeros(n, dtype=torch.float64, device="cuda")
    F, gW = torch.zeros((n, 3), dtype=torch.float64, device="cuda"), torch.zeros_like(W)
    w3 = torch.zeros((S.nst, 3, 3), dtype=torch.float64, device="cuda")
    for i, j, sh in S.pairs(rc3, 8192):
        cnt = torch.bincount(i - i[0], minlength=int(i[-1] - i[0]) + 1)
        start = torch.cumsum(cnt, 0) - cnt
        own = cnt[i - i[0]]
        p = torch.arange(len(i), device="cuda")
        a = p.repeat_interleave(own)  # every ordered pair of list entries of one atom
        first = (torch.cumsum(own, 0) - own).repeat_interleave(own)
        b = start[i[a] - i[0]] + torch.arange(len(a), device="cuda") - first
        k = ((a < b) & (((x[j[b]] + sh[b]) - (x[j[a]] + sh[a])).pow(2).sum(1) < rc3 * rc3)).nonzero().squeeze(1)
        a, b = a[k], b[k]
        vi, vj, vk = i[a], j[a], j[b]
        with torch.enable_grad():
            xs = x.detach().requires_grad_(True)
            Wl = W.detach().requires_grad_(True)
            eps = torch.zeros((S.nst, 3, 3), dtype=torch.float64, device="cuda", requires_grad=True)

            def vec(d):
                return d + (d.unsqueeze(1) @ eps[S.sid[vi]]).squeeze(1)
            u, w = vec(xs[vj] + sh[a] - xs[vi]), vec(xs[vk] + sh[b] - xs[vi])
            X, Y, Z = u.pow(2).sum(1), w.pow(2).sum(1), (w - u).pow(2).sum(1)

            def c6(p_, q_):
                return torch.einsum("na,nab,nb->n", Wl[p_], c6r[t[p_], t[q_]], Wl[q_])

            def rad(p_, q_):
                return theta[2] * (3.0 * sq[t[p_]] * sq[t[q_]]).sqrt() + theta[3]
            pr = X * Y * Z
            ang = (1.0 + 0.375 * (X + Y - Z) * (X + Z - Y) * (Y + Z - X) / pr) / pr ** 1.5
            q = (rad(vi, vj) * rad(vi, vk) * rad(vj, vk) / pr.sqrt()) ** third
            e = prm["s9"] * (c6(vi, vj) * c6(vi, vk) * c6(vj, vk)).sqrt() * ang / (1.0 + 6.0 * q) / 3.0
            gx, gw, ge = torch.autograd.grad(e.sum(), (xs, Wl, eps))
        U = U + _add(n, vi, e.detach())
        F, gW, w3 = F - gx, gW + gw, w3 - ge
    return U, F, w3, (gW * dW).sum(1)


def _exact_batch(case, b, prm, pos=None, **kw):
    S = _System(b.pos if pos is None else pos, b.types, b.offsets, b.cells, b.pbc,
                max(prm["rc_disp"], prm["rc_cn"]) / BOHR)
    theta = torch.tensor([prm[k] for k in ("s6", "s8", "a1", "a2")], dtype=torch.float64, device="cuda")
    return S, theta, _d3_64(S, b.tables, prm, S.x, theta, **kw)


def _exact_refit(case, b, prm, seed):
    from torch.autograd import forward_ad as fwad
    S, theta, o = _exact_batch(case, b, prm)
    e, f = _targets(b, seed)
    with torch.enable_grad():
        E, F = o["E"].clone().requires_grad_(True), o["F"].clone().requires_grad_(True)
        n = torch.tensor(np.diff(b.offsets).astype(np.float64), device="cuda")
        gE, gF = torch.autograd.grad(_loss(E, F, torch.tensor(e, device="cuda"), torch.tensor(f, device="cuda"), n),
                                     (E, F))

    def along(dx, dth):  # the derivative of (E, F) along a direction of positions (A) or parameters
        with fwad.dual_level():
            x = fwad.make_dual(S.x, dx / BOHR) if dx is not None else S.x
            th = fwad.make_dual(theta, dth) if dth is not None else theta
            r = _d3_64(S, b.tables, prm, x, th)
            return [fwad.unpack_dual(r[k]).tangent for k in ("E", "F")]
    hv = along(gF, None)[1]  # the Hessian is symmetric: J^T gF = J gF
    dpos = -gE[S.sid][:, None] * o["F"] + hv
    dth = []
    for k in range(4):
        u = torch.zeros(4, dtype=torch.float64, device="cuda")
        u[k] = 1.0
        tE, tF = along(None, u)
        dth.append((gE * tE).sum() + (gF * tF).sum())
    return dict(E=o["E"], F=o["F"], dpos=dpos, dtheta=torch.stack(dth))


@torch.no_grad()
def exact(case, seed):
    kind = case["kind"]
    b = _batch(case, seed)
    prm = _params(case)
    if kind == "refit":
        return _exact_refit(case, b, prm, seed)
    if kind == "heat":
        _, _, o = _exact_batch(case, b, prm, parts=True)
        vel = torch.tensor(wl.maxwell_velocities(wl.atom_masses(b), 300.0, seed), device="cuda")
        return dict(E=o["E"], F=o["F"], W=o["W"], w_atom=o["w_atom"], J=(o["w_atom"] @ vel.unsqueeze(-1)).squeeze(-1))
    _, _, o = _exact_batch(case, b, prm, site=bool(case.get("atoms")))
    r = dict(E=o["E"], F=o["F"], W=o["W"])
    if kind in ("call", "npt"):
        r["W"] = o["W"][0]
    if case.get("atoms"):
        r.update(e_atom=o["e_atom"], cn=o["cn"])
    return r
