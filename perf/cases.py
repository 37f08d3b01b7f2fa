"""Performance cases of the imaginary-time GW calls, through the public entry points.

A case is one call (or, for "g0w0", the chain of calls) that a program of this
library makes: chi(i tau) in each precision form, the screening chain, the
diagonal, batched and full-matrix self-energies.  Systems carry the per-atom
basis of the other workloads of this repository ('C': 13 primary and 30 RI
functions, 'H': 5 and 12); the three-centre blocks are normal deviates times
exp(-0.5 r_AB^2) exp(-0.8 r_mid,P), the orbitals eigenvectors of a banded
Hamiltonian with a 0.3 Ha gap, the tau points log-spaced in [0.01, 50] a.u.
"""

import math

import numpy as np
import torch

from paper_2104_09857_gb300 import Context, PRECISIONS, _lib

BASIS = {"C": (13, 30), "H": (5, 12)}
GAP, WIDTH = 0.3, 2.3


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest calls: every tau point of one ring molecule, nothing filtered
        {"name": "chi fp64 ring-12", "call": "chi", "shape": "ring", "atoms": 12, "form": "fp64", "thr": 0.0, "taus": 10},
        {"name": "chi fp16x3 ring-12", "call": "chi", "shape": "ring", "atoms": 12, "form": "fp16x3", "thr": 0.0, "taus": 10},
        # plain FP64 chi of a short ribbon: the form that the mixed ones are judged by
        {"name": "chi fp64 ribbon-40", "call": "chi", "shape": "ribbon", "atoms": 40, "form": "fp64", "thr": 1e-9, "taus": 1},
        # the FP32 form on the CUDA cores
        {"name": "chi fp32 ribbon-58", "call": "chi", "shape": "ribbon", "atoms": 58, "form": "fp32", "thr": 1e-9, "taus": 1},
        # the production form: an ordinary and a large ribbon
        {"name": "chi fp16x3 ribbon-58", "call": "chi", "shape": "ribbon", "atoms": 58, "form": "fp16x3", "thr": 1e-9, "taus": 4},
        {"name": "chi fp16x3 ribbon-118", "call": "chi", "shape": "ribbon", "atoms": 118, "form": "fp16x3", "thr": 1e-9, "taus": 1},
        # the six-product form on a compact disordered cluster (ragged windows, mixed species)
        {"name": "chi bf16x6 cluster-45", "call": "chi", "shape": "cluster", "atoms": 45, "form": "bf16x6", "thr": 1e-9, "taus": 2},
        # chi(i tau) -> W^c(i tau), FP64 throughout
        {"name": "chi_to_w ribbon-58", "call": "chi_to_w", "shape": "ribbon", "atoms": 58, "form": "fp64", "thr": 0.0, "taus": 6},
        # HOMO and LUMO self-energy of one molecule in FP64
        {"name": "sigma fp64 ribbon-58", "call": "sigma", "shape": "ribbon", "atoms": 58, "form": "fp64", "thr": 1e-9, "taus": 6},
        # many molecules of uneven size in one call
        {"name": "sigma batch fp16x3 12 molecules", "call": "sigma_batch", "shape": "ring", "atoms": 90, "form": "fp16x3", "thr": 1e-9, "taus": 4, "molecules": 12},
        # the full AO matrix of the self-energy of a molecule
        {"name": "sigma_ao ribbon-28", "call": "sigma_ao", "shape": "ribbon", "atoms": 28, "form": "fp64", "thr": 1e-9, "taus": 2},
        # a whole G0W0 pass (without the quasiparticle solve) of a small molecule
        {"name": "g0w0 fp16x3 ring-24", "call": "g0w0", "shape": "ring", "atoms": 24, "form": "fp16x3", "thr": 1e-9, "taus": 8},
    ]


# largest atom counts at one tau point that stay below the largest listed case
MOST_ATOMS = {"fp64": 40, "fp32": 58, "bf16x3": 110, "bf16x6": 90, "fp16x3": 110}


def draw(rng):
    def between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["chi", "chi", "chi", "chi", "chi_to_w", "sigma", "sigma_batch", "sigma_ao", "g0w0"])
    shape = rng.choice(["ring", "ribbon", "ribbon", "cluster"])
    thr = rng.choice([0.0, 1e-9, 1e-9, 1e-6])
    form = "fp64"
    if call == "chi":
        form = rng.choice(["fp64", "fp32", "bf16x3", "bf16x6", "fp16x3", "fp16x3"])
        most = min(MOST_ATOMS[form], 24 if thr == 0.0 else 60 if shape == "cluster" else 200)
        atoms = between(5, most)
        # chi's work grows with the fourth power of a small system's size
        taus = max(1, min(10, int((most / atoms) ** 3)))
        return {"call": call, "shape": shape, "atoms": atoms, "form": form, "thr": thr, "taus": rng.randint(1, taus)}
    if call == "chi_to_w":
        return {"call": call, "shape": shape, "atoms": between(6, 60), "form": form, "thr": 0.0, "taus": rng.randint(4, 6)}
    if call == "sigma":
        form = rng.choice(["fp64", "fp16x3", "bf16x6"])
        return {"call": call, "shape": shape, "atoms": between(6, 24 if thr == 0.0 else 60), "form": form, "thr": thr, "taus": rng.randint(2, 8)}
    if call == "sigma_batch":
        return {"call": call, "shape": "ring", "atoms": between(20, 90), "form": rng.choice(["fp16x3", "bf16x6"]), "thr": 1e-9,
                "taus": rng.randint(1, 4), "molecules": rng.randint(3, 12)}
    if call == "sigma_ao":
        return {"call": call, "shape": shape, "atoms": between(5, 28), "form": form, "thr": thr, "taus": rng.randint(1, 2)}
    return {"call": call, "shape": shape, "atoms": between(6, 24), "form": rng.choice(["fp64", "fp16x3"]), "thr": 1e-9, "taus": rng.randint(6, 8)}


# ---------------------------------------------------------------------------
# systems
# ---------------------------------------------------------------------------
def geometry(shape, n):
    """(positions [n, 3] in Angstrom, species) of n atoms."""
    if shape == "ring":  # carbons 1.4 A apart on a circle, a hydrogen outside every other one
        nc = n - n // 3
        radius = 1.4 / (2 * math.sin(math.pi / max(nc, 3)))
        at = [(radius, 2 * math.pi * k / nc, "C") for k in range(nc)]
        at += [(radius + 1.09, 2 * math.pi * (2 * k % nc) / nc, "H") for k in range(n - nc)]
        xyz = [(r * math.cos(a), r * math.sin(a), 0.0) for r, a, _ in at]
        return np.array(xyz), [s for _, _, s in at]
    if shape == "ribbon":  # four dimer lines of an armchair ribbon with hydrogens along both edges
        dy, top, at = 1.4 * math.sqrt(0.75), 3 * 1.4 * math.sqrt(0.75), []
        for cell in range(n // 12 + 2):
            for k in range(4):
                for x in ((0.0, 1.4) if k % 2 == 0 else (2.1, 3.5)):
                    at.append((4.2 * cell + x, k * dy, "C"))
            at += [(4.2 * cell - 0.5, -0.95, "H"), (4.2 * cell + 1.9, -0.95, "H")]
            at += [(4.2 * cell + 1.6, top + 0.95, "H"), (4.2 * cell + 4.0, top + 0.95, "H")]
        at = sorted(at)[:n]
        return np.array([(x, y, 0.0) for x, y, _ in at]), [s for _, _, s in at]
    # cluster: uniform positions at 0.1 atoms per cubic Angstrom, at least 1 A apart
    rng, box, xyz = np.random.RandomState(1000 + n), (n / 0.1) ** (1 / 3), []
    while len(xyz) < n:
        p = rng.uniform(0, box, 3)
        if all(np.linalg.norm(p - q) >= 1.0 for q in xyz):
            xyz.append(p)
    return np.array(xyz), ["C" if u < 2 / 3 else "H" for u in rng.uniform(size=n)]


class System:
    def __init__(self, shape, n):
        self.xyz, species = geometry(shape, n)
        self.n_ao = np.array([BASIS[s][0] for s in species], dtype=np.int32)
        self.n_ri = np.array([BASIS[s][1] for s in species], dtype=np.int32)
        self.nao, self.nri = int(self.n_ao.sum()), int(self.n_ri.sum())
        self.n_occ = min(self.nao - 1, sum(6 if s == "C" else 1 for s in species) // 2)

    def blocks(self, thr):
        """([n, 3] atoms (A, B, P) of the stored blocks, A <= B, their scales and sizes):
        those with an expected norm of thr or more."""
        x, n = self.xyz, len(self.n_ao)
        a, b = np.triu_indices(n)
        mid = 0.5 * (x[a] + x[b])
        r_ab = np.sum((x[a] - x[b]) ** 2, axis=1)
        r_mp = np.sqrt(np.sum((mid[:, None] - x[None]) ** 2, axis=2))
        scale = np.exp(-0.5 * r_ab)[:, None] * np.exp(-0.8 * r_mp)
        size = (self.n_ao[a] * self.n_ao[b])[:, None].astype(np.int64) * self.n_ri[None]
        pair, p = np.nonzero(scale * np.sqrt(size) >= thr)
        return np.stack([a[pair], b[pair], p], axis=1).astype(np.int32), scale[pair, p], size[pair, p]


def tensor(system, thr, seed):
    """(blocks, values on the GPU) of the three-centre tensor."""
    blk, scale, size = system.blocks(thr)
    off = np.concatenate([[0], np.cumsum(size)])
    gen = torch.Generator("cuda").manual_seed(seed)
    data = torch.randn(int(off[-1]), dtype=torch.float64, device="cuda", generator=gen)
    scale_d, size_d = torch.from_numpy(scale).cuda(), torch.from_numpy(size).cuda()
    b0 = 0
    while b0 < len(size):  # runs of blocks, so that the index arrays stay small
        b1 = max(b0 + 1, int(np.searchsorted(off, off[b0] + (1 << 26), side="right")) - 1)
        data[off[b0]:off[b1]] *= torch.repeat_interleave(scale_d[b0:b1], size_d[b0:b1])
        b0 = b1
    na, npf = system.n_ao[blk[:, 0]], system.n_ri[blk[:, 2]]
    for va, vp in ((13, 30), (13, 12), (5, 30), (5, 12)):  # (A, A, P) blocks are symmetric
        at = np.nonzero((blk[:, 0] == blk[:, 1]) & (na == va) & (npf == vp))[0]
        if len(at):
            pos = torch.from_numpy(off[at]).cuda()[:, None] + torch.arange(va * va * vp, device="cuda")
            v = data[pos].reshape(-1, va, va, vp)
            data[pos] = (0.5 * (v + v.transpose(1, 2))).reshape(len(at), -1)
    return blk, data


def orbitals(system, seed):
    rng = np.random.RandomState((seed * 7919 + 17) % (1 << 32))
    r = np.linalg.norm(system.xyz[:, None] - system.xyz[None], axis=2)
    env = np.repeat(np.repeat(np.where(r <= 5.0, np.exp(-r), 0.0), system.n_ao, axis=0), system.n_ao, axis=1)
    h = rng.standard_normal((system.nao, system.nao)) * env
    w, c = np.linalg.eigh(h + h.T)
    w, k = w * ((WIDTH - GAP) / (w[-1] - w[0])), system.n_occ
    eps = np.concatenate([w[:k] - w[k - 1] - GAP / 2, w[k:] - w[k] + GAP / 2])
    return np.ascontiguousarray(c), eps


def tau_grid(n):
    return 0.01 * 5000.0 ** (np.arange(n) / max(n - 1, 1)) if n > 1 else np.array([1.0])


def transforms(tau):
    """Least-squares cosine-transform weights gamma [omega][tau], delta [tau][omega]."""
    n = len(tau)
    omega = 0.5 * GAP * (4 * WIDTH / GAP) ** (np.arange(n) / max(n - 1, 1))
    x = GAP * (WIDTH / GAP) ** (np.arange(200) / 199)
    e = np.exp(-np.outer(x, tau))
    f = 2 * x[:, None] / (x[:, None] ** 2 + omega[None] ** 2)
    gamma = np.linalg.lstsq(e, f, rcond=1e-4)[0].T
    delta = np.linalg.lstsq(f, e, rcond=1e-4)[0].T
    return np.ascontiguousarray(gamma), np.ascontiguousarray(delta)


def coulomb(system):
    c = np.repeat(system.xyz, system.n_ri, axis=0)
    v = 1.0 / np.sqrt(np.sum((c[:, None] - c[None]) ** 2, axis=2) + 1.0)
    return v + np.eye(system.nri)


def response(nri, tau, rate, seed):
    """[n_tau, nri, nri] of the sign and decay of chi(i tau) or W^c(i tau): minus a
    random positive semidefinite matrix falling as exp(-rate tau)."""
    gen = torch.Generator("cuda").manual_seed(seed + 5)
    r = torch.randn(nri, nri, dtype=torch.float64, device="cuda", generator=gen)
    a = -(r @ r.T) / nri
    a = 0.5 * (a + a.T)
    return torch.stack([a * math.exp(-rate * float(t)) for t in tau])


def sizes(case):
    """Atom counts of the case's molecules (one, but for the batch)."""
    m = case.get("molecules", 1)
    return [case["atoms"]] if m == 1 else [10 + (case["atoms"] - 10) * i // (m - 1) for i in range(m)]


def frontier(system):
    return [system.n_occ - 1, system.n_occ]


# ---------------------------------------------------------------------------
# preparation and the timed call
# ---------------------------------------------------------------------------
def prepare(case, seed):
    tau = tau_grid(case["taus"])
    state = {"case": case, "tau": tau, "members": []}
    for i, n in enumerate(sizes(case)):
        system = System(case["shape"], n)
        ctx = Context(0)
        ctx.set_basis(system.xyz, system.n_ao, system.n_ri)
        if case["call"] != "chi_to_w":
            blk, data = tensor(system, case["thr"], seed + 101 * i)
            ctx.set_3c_tensor(blk, data.cpu().numpy())
        c, eps = orbitals(system, seed + 101 * i)
        ctx.set_greens(c, eps, system.n_occ, 0.0, tau)
        state["members"].append((system, ctx))
    call, (system, ctx) = case["call"], state["members"][0]
    if call in ("chi_to_w", "g0w0"):
        state["gamma"], state["delta"] = transforms(tau)
        state["v"] = coulomb(system)
        if call == "chi_to_w":
            state["chi"] = response(system.nri, tau, 0.3, seed)
        else:
            state["v"] *= 0.01
    elif call == "sigma_batch":
        state["w"] = [response(s.nri, tau, 0.1, seed + 7 * i).cpu().numpy() for i, (s, _) in enumerate(state["members"])]
    elif call == "sigma":
        state["w"] = response(system.nri, tau, 0.1, seed)
    elif call == "sigma_ao":
        state["w"] = response(system.nri, tau, 0.1, seed).cpu().numpy()
    return state


def run(state):
    case, (system, ctx) = state["case"], state["members"][0]
    call, form, thr = case["call"], case["form"], case["thr"]
    if call == "chi":
        return ctx.chi_tau(thr, form)
    if call == "chi_to_w":
        return ctx.chi_to_w(state["chi"], state["v"], state["gamma"], state["delta"])
    if call == "sigma":
        return ctx.sigma_tau(state["w"], frontier(system), thr, form)
    if call == "sigma_batch":
        return _lib.gw_sigma_tau_batch([c.ctx for _, c in state["members"]], state["w"], [frontier(s) for s, _ in state["members"]],
                                       thr, PRECISIONS[form])
    if call == "sigma_ao":
        return _lib.gw_sigma_ao_tau(ctx.ctx, state["w"], len(state["tau"]), system.nao, thr)
    chi = ctx.chi_tau(thr, form)
    w = ctx.chi_to_w(chi, state["v"], state["gamma"], state["delta"])
    return {"chi": chi, "w": w, "sigma": ctx.sigma_tau(w, frontier(system), thr, form)}


def work(case):
    """Reads and writes of the stored blocks, matrices and results once per pass; flops of
    the atom-block products that the stored blocks leave (chi's upper triangle only)."""
    nt, call = case["taus"], case["call"]
    flops = bytes_ = 0.0
    for n in sizes(case):
        s = System(case["shape"], n)
        ao, ri = float(s.nao), float(s.nri)
        if call != "chi_to_w":
            blk, _, size = s.blocks(case["thr"])
            both = float(np.sum(np.where(blk[:, 0] == blk[:, 1], 1, 2) * size))
            reach = np.zeros((n, n), dtype=bool)  # RI atoms that each atom shares a block with
            reach[blk[:, 0], blk[:, 2]] = reach[blk[:, 1], blk[:, 2]] = True
            win = float(np.sum(s.n_ao * (reach @ s.n_ri)))
            bytes_ += 8 * float(size.sum())
        if call in ("chi", "g0w0"):
            flops += nt * (4 * ao * both + win * win + 2 * ao * ao * ao)
            bytes_ += 8 * (nt * ri * ri + ao * ao)
        if call in ("chi_to_w", "g0w0"):
            flops += nt * (25 / 3 * ri ** 3 + 4 * nt * ri * ri) + ri ** 3 / 3
            bytes_ += 8 * (2 * nt + 1) * ri * ri
        if call in ("sigma", "sigma_batch", "g0w0"):
            flops += 2 * (2 * both + nt * 2 * (ao * ri * ri + ao * ao * ri + 2 * ao * ao)) + nt * 2 * ao ** 3
            bytes_ += 8 * (nt * ri * ri + ao * ao)
        if call == "sigma_ao":
            flops += nt * (2 * ao * ao * ri * ri + 8 * ao ** 3 * ri + 2 * ao ** 3)
            bytes_ += 8 * nt * (ri * ri + 2 * ao * ao)
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ---------------------------------------------------------------------------
class Dense:
    """Dense tensors of one molecule and the definitions of its results."""

    def __init__(self, case, n, seed):
        self.s, self.thr = System(case["shape"], n), case["thr"]
        s = self.s
        self.ind_ao, self.ind_ri = (torch.from_numpy(np.repeat(np.eye(len(k)), k, axis=1)).cuda() for k in (s.n_ao, s.n_ri))
        c, eps = orbitals(s, seed)
        self.c, self.eps = torch.from_numpy(c).cuda(), torch.from_numpy(eps).cuda()
        if case["call"] != "chi_to_w":
            self.t = self.expand(*tensor(s, self.thr, seed))

    def expand(self, blk, data):
        s = self.s
        ao, ri = (np.concatenate([[0], np.cumsum(k)]) for k in (s.n_ao, s.n_ri))
        t = torch.zeros(s.nao, s.nao, s.nri, dtype=torch.float64, device="cuda")
        size = s.n_ao[blk[:, 0]].astype(np.int64) * s.n_ao[blk[:, 1]] * s.n_ri[blk[:, 2]]
        off = np.concatenate([[0], np.cumsum(size)])
        kind = s.n_ao[blk[:, 0]] * 10000 + s.n_ao[blk[:, 1]] * 100 + s.n_ri[blk[:, 2]]
        for k in np.unique(kind):
            na, nb, npf = int(k) // 10000, int(k) // 100 % 100, int(k) % 100
            for at in np.array_split(np.nonzero(kind == k)[0], 1 + int(np.sum(kind == k)) // 20000):
                v = data[torch.from_numpy(off[at]).cuda()[:, None] + torch.arange(na * nb * npf, device="cuda")]
                v = v.reshape(-1, na, nb, npf)
                v = torch.where((v.square().sum((1, 2, 3), keepdim=True).sqrt() < self.thr), 0.0, v)
                i, j, p = (torch.from_numpy(o[blk[at, x]]).cuda()[:, None] + torch.arange(m, device="cuda")
                           for o, x, m in ((ao, 0, na), (ao, 1, nb), (ri, 2, npf)))
                t[i[:, :, None, None], j[:, None, :, None], p[:, None, None, :]] = v
                t[j[:, :, None, None], i[:, None, :, None], p[:, None, None, :]] = v.transpose(1, 2)
        return t

    def drop(self, x, kinds):
        """x with its atom blocks of norm below thr set to zero; an axis is 'a' (primary) or 'r' (RI)."""
        if self.thr == 0.0:
            return x
        sq, ind = x * x, {"a": self.ind_ao, "r": self.ind_ri}
        for axis, k in enumerate(kinds):
            sq = torch.movedim(torch.tensordot(ind[k], sq, dims=([1], [axis])), 0, axis)
        keep = sq.sqrt() >= self.thr
        for axis, k in enumerate(kinds):
            keep = keep.index_select(axis, ind[k].argmax(0))
        return torch.where(keep, x, 0.0)

    def greens(self, tau):
        k, half = self.s.n_occ, torch.exp(0.5 * tau * -self.eps.abs())
        o, v = self.c[:, :k] * half[:k], self.c[:, k:] * half[k:]
        return self.drop(o @ o.T, "aa"), self.drop(v @ v.T, "aa")

    def chi(self, tau):
        s, out = self.s, []
        atom = self.ind_ri.argmax(0)
        for t in tau:
            go, gv = self.greens(float(t))
            m = self.drop((go @ self.t.reshape(s.nao, -1)).reshape(s.nao, s.nao, s.nri), "aar")
            n = self.drop(torch.matmul(gv, self.t), "aar")
            x = -(m.reshape(-1, s.nri).T @ n.reshape(-1, s.nri))
            out.append(torch.where(atom[:, None] > atom[None], x.T, x))
        return torch.stack(out)

    def sigma(self, w, tau):
        out = torch.zeros(2, len(tau), 2, dtype=torch.float64)
        for a, orb in enumerate(frontier(self.s)):
            b = self.drop(torch.tensordot(self.c[:, orb], self.t, dims=([0], [0])), "ar")
            for j, t in enumerate(tau):
                z = b @ w[j] @ b.T
                for k, g in enumerate(self.greens(float(t))):
                    out[a, j, k] = float((g * z).sum()) * (1 if k else -1)
        return out

    def sigma_ao(self, w, tau):
        s, out = self.s, torch.zeros(len(tau), 2, self.s.nao, self.s.nao, dtype=torch.float64)
        for j, t in enumerate(tau):
            z = torch.matmul(self.t, w[j]).reshape(s.nao, -1)
            for k, g in enumerate(self.greens(float(t))):
                u = (g @ z).reshape(s.nao, s.nao, s.nri).transpose(0, 1).reshape(s.nao, -1)
                out[j, k] = (self.t.reshape(s.nao, -1) @ u.T).cpu() * (1 if k else -1)
        return out


def screened(chi, v, gamma, delta):
    v, low = torch.from_numpy(v).cuda(), torch.linalg.cholesky(torch.from_numpy(v).cuda())
    one = torch.eye(len(v), dtype=torch.float64, device="cuda")
    w = torch.zeros_like(chi)
    for k in range(len(gamma)):
        x = sum(float(g) * chi[j] for j, g in enumerate(gamma[k]))
        eps = one - low.T @ x @ low
        wk = low @ (torch.cholesky_solve(low.T.contiguous(), torch.linalg.cholesky(eps)) - low.T)
        for j in range(len(chi)):
            w[j] += float(delta[j, k]) * wk
    return w


def exact(case, seed):
    call, tau = case["call"], tau_grid(case["taus"])
    s = System(case["shape"], sizes(case)[0])
    if call == "chi" and case["taus"] * (s.nao * s.nri) ** 2 > 8e12:
        return None  # dense products of more than some 20 s
    if call == "chi_to_w":
        return screened(response(s.nri, tau, 0.3, seed), coulomb(s), *transforms(tau))
    if call == "sigma_batch":
        out = []
        for i, n in enumerate(sizes(case)):
            d = Dense(case, n, seed + 101 * i)
            out.append(d.sigma(response(d.s.nri, tau, 0.1, seed + 7 * i), tau))
            del d
        return out
    d = Dense(case, sizes(case)[0], seed)
    if call == "chi":
        return d.chi(tau)
    if call == "g0w0":
        chi = d.chi(tau)
        w = screened(chi, 0.01 * coulomb(s), *transforms(tau))
        return {"chi": chi, "w": w, "sigma": d.sigma(w, tau)}
    w = response(s.nri, tau, 0.1, seed)
    return d.sigma(w, tau) if call == "sigma" else d.sigma_ao(w, tau)
