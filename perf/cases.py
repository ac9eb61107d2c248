"""Performance cases of the dense Kohn-Sham solver: what a program that uses this package
asks of it, through the public entry points (Handle, autograd), over the range of sizes,
precisions and options in use.

The matrices are localized-basis Kohn-Sham matrices: a random 3D cluster (0.01 atoms/bohr^3,
15 functions per atom) or a 1D chain (spacing 2 bohr, 8 functions per atom), with
O_ij = 0.3 exp(-d/1.5) u_ij, H_ij = -0.5 exp(-d/1.2) (1 + 0.1 g_ij), H_ii ~ U(-1, 0.5) and
S = I + alpha O scaled so that lambda_min(S) >= about 1e-2. A cluster with integer occupation
is an insulator (as integer occupation is used for): one function per atom lies lower, which
opens a gap of about 0.3 Ha above two occupied states per atom. The matrices are made on the
GPU from the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1705_11191_gb300 as egb
from paper_1705_11191_gb300 import autograd as ega

KT = 0.01        # Fermi-Dirac width (Ha)
CUTOFF = 12.0    # bohr: the sparse pattern's interaction range
EXACT_MAX = 5200  # largest (real-form) order that the 64-bit reference solves quickly


def listed():
    return [
        # one small molecule, binary64: every call is launches and serial chains
        {"name": "dm-f64-n120", "kind": "dm", "prec": "f64", "geom": "cluster", "n": 120, "kt": 0.0, "full": False},
        # the 64-atom chain, all 512 states computed, integer occupation
        {"name": "dm-f64-chain-n512", "kind": "dm", "prec": "f64", "geom": "chain", "n": 512, "kt": 0.0, "full": True},
        # a medium metal-like system in binary64, odd size, smeared occupation
        {"name": "dm-f64-n1531", "kind": "dm", "prec": "f64", "geom": "cluster", "n": 1531, "kt": KT, "full": False},
        # a large system in binary64 (the route of highest accuracy)
        {"name": "dm-f64-n5000", "kind": "dm", "prec": "f64", "geom": "cluster", "n": 5000, "kt": 0.0, "full": False},
        # the SCF step of a small system on the binary32 + refinement route, ragged size
        {"name": "dm-refine-n777", "kind": "dm", "prec": "refine", "geom": "cluster", "n": 777, "kt": KT, "full": False},
        # the same for a medium system
        {"name": "dm-refine-n4096", "kind": "dm", "prec": "refine", "geom": "cluster", "n": 4096, "kt": KT, "full": False},
        # the headline problem: n = 16384, 2048 states
        {"name": "dm-refine-n16384", "kind": "dm", "prec": "refine", "geom": "cluster", "n": 16384, "kt": 0.0, "full": False},
        # complex Hermitian k-points of one cell with one chemical potential
        {"name": "kpoints-refine-8x1000", "kind": "kpoints", "prec": "refine", "n": 1000, "nprob": 8},
        # real problems of uneven size, each with its own chemical potential
        {"name": "mixed-refine-12", "kind": "mixed", "prec": "refine", "lo": 256, "hi": 2048, "nprob": 12, "draws": 4},
        # differentiable free energy: forward solve and dF/dH, dF/dS
        {"name": "free-energy-grad-n2000", "kind": "fgrad", "prec": "refine", "n": 2000},
        # differentiable eigenpairs: all of them, and the adjoint of a loss on the occupied ones
        {"name": "eigen-grad-f64-n600", "kind": "egrad", "prec": "f64", "n": 600},
        # sparse (CSC) input and output, a long chain
        {"name": "csc-f64-n1000", "kind": "csc", "prec": "f64", "n": 1000},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dm64", "dm32", "dm32", "kpoints", "mixed", "fgrad", "egrad", "csc"])
    if kind == "dm64":
        return {"kind": "dm", "prec": "f64", "geom": rng.choice(["cluster", "chain"]),
                "n": _logint(rng, 64, 5000), "kt": rng.choice([0.0, KT]), "full": False}
    if kind == "dm32":
        kt = rng.choice([0.0, KT])
        return {"kind": "dm", "prec": "refine", "geom": "cluster",
                "n": _logint(rng, 500, 14000 if kt == 0.0 else 5000), "kt": kt, "full": False}
    if kind == "kpoints":
        return {"kind": "kpoints", "prec": "refine", "n": _logint(rng, 256, 1200), "nprob": rng.randint(4, 16)}
    if kind == "mixed":
        return {"kind": "mixed", "prec": "refine", "lo": 256, "hi": rng.randint(600, 2500),
                "nprob": rng.randint(6, 14), "draws": rng.randint(0, 999)}
    if kind == "fgrad":
        return {"kind": "fgrad", "prec": "refine", "n": _logint(rng, 500, 4000)}
    if kind == "egrad":
        return {"kind": "egrad", "prec": "f64", "n": _logint(rng, 100, 1000)}
    return {"kind": "csc", "prec": "f64", "n": _logint(rng, 300, 3000)}


# ---------------------------------------------------------------- inputs
def _positions(rng, n_atoms):
    """Uniform in a cube, 2 bohr minimum separation."""
    side = (n_atoms / 0.01) ** (1.0 / 3.0)
    pos = np.zeros((n_atoms, 3))
    k = 0
    while k < n_atoms:
        p = rng.random(3) * side
        if k == 0 or np.min(np.sum((pos[:k] - p) ** 2, axis=1)) >= 4.0:
            pos[k] = p
            k += 1
    return pos, side


def _lambda_min(o, steps=96):
    """A lower bound, to about its residual, of the smallest eigenvalue (Lanczos)."""
    n = o.shape[0]
    steps = min(steps, n)
    v = torch.ones(n, 1, dtype=o.dtype, device=o.device) + 0.1 * torch.sin(
        torch.arange(n, dtype=torch.float64, device=o.device))[:, None]
    basis = torch.zeros((n, steps + 1), dtype=o.dtype, device=o.device)
    basis[:, :1] = v / torch.linalg.vector_norm(v)
    al, be = [], []
    for j in range(steps):
        q = basis[:, :j + 1]
        w = o @ q[:, j:]
        al.append((q[:, j:].conj() * w).sum().real)
        w = w - q @ (q.conj().T @ w)
        w = w - q @ (q.conj().T @ w)
        be.append(torch.linalg.vector_norm(w))
        basis[:, j + 1:j + 2] = w / be[-1].clamp_min(1e-300)
    t = torch.diag(torch.stack(al))
    if steps > 1:
        off = torch.stack(be[:-1])
        t = t + torch.diag(off, 1) + torch.diag(off, -1)
    val, vec = torch.linalg.eigh(t)
    return float(val[0] - be[-1] * vec[-1, 0].abs() - 1e-6)


def _overlap(o):
    lam = _lambda_min(o)
    s = o * (1.0 if 1.0 + lam >= 1e-2 else (1.0 - 1e-2) / (-lam))
    s.diagonal().fill_(1.0)
    return s


def _real_problem(n, seed, geom, cutoff=None, gap=False):
    """(H, S, mask or None), symmetric float64 (n, n) CUDA tensors."""
    dev = torch.device("cuda")
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=dev).manual_seed(int(rng.integers(1 << 60)))
    per = 8 if geom == "chain" else 15
    n_atoms = -(-n // per)
    if geom == "chain":
        pos = np.zeros((n_atoms, 3))
        pos[:, 0] = 2.0 * np.arange(n_atoms)
    else:
        pos, _ = _positions(rng, n_atoms)
    xyz = torch.from_numpy(pos[np.arange(n) // per]).to(dev)
    d2 = torch.zeros((n, n), dtype=torch.float64, device=dev)
    for c in range(3):
        d2 += (xyz[:, c, None] - xyz[None, :, c]) ** 2
    d = d2.sqrt_()
    mask = None if cutoff is None else (d <= cutoff)
    u = torch.rand((n, n), dtype=torch.float64, device=dev, generator=gen)
    o = torch.triu(u.mul_(0.3).mul_(torch.exp(d / -1.5)), 1)
    if mask is not None:
        o *= mask
    o = o + o.T
    s = _overlap(o)
    del u, o
    g = torch.randn((n, n), dtype=torch.float64, device=dev, generator=gen)
    h = torch.triu(g.mul_(0.1).add_(1.0).mul_(-0.5).mul_(torch.exp(d / -1.2)), 1)
    if mask is not None:
        h *= mask
    del g, d, d2
    h = h + h.T
    r = torch.rand(n, dtype=torch.float64, device=dev, generator=gen)
    hd = r * 1.5 - (0.5 if gap else 1.0)
    if gap:
        hd[::per] = r[::per] * 0.5 - 1.5
    h.diagonal().copy_(hd)
    return h, s, mask


def _kpoint_problems(n, nprob, seed):
    """Hermitian H(k), S(k) of one cell (27 lattice blocks) at nprob points of a shifted line
    grid through the Brillouin zone; complex128 (n, n) CUDA tensors."""
    dev = torch.device("cuda")
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=dev).manual_seed(int(rng.integers(1 << 60)))
    n_atoms = -(-n // 15)
    pos, side = _positions(rng, n_atoms)
    xyz = torch.from_numpy(pos[np.arange(n) // 15]).to(dev)
    ks = [((p + 0.25) / nprob, ((3 * p) % nprob + 0.25) / nprob, ((7 * p) % nprob + 0.25) / nprob)
          for p in range(nprob)]
    hk = [torch.zeros((n, n), dtype=torch.complex128, device=dev) for _ in ks]
    ok = [torch.zeros((n, n), dtype=torch.complex128, device=dev) for _ in ks]
    cells = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]
    for R in cells[:14]:  # R and -R together; the last one is the home cell
        d2 = torch.zeros((n, n), dtype=torch.float64, device=dev)
        for c in range(3):
            d2 += (xyz[:, c, None] - xyz[None, :, c] - side * R[c]) ** 2
        d = d2.sqrt_()
        u = torch.rand((n, n), dtype=torch.float64, device=dev, generator=gen)
        g = torch.randn((n, n), dtype=torch.float64, device=dev, generator=gen)
        o_r = 0.3 * torch.exp(d / -1.5) * u
        h_r = -0.5 * torch.exp(d / -1.2) * (1.0 + 0.1 * g)
        if R == (0, 0, 0):
            o_r, h_r = torch.triu(o_r, 1), torch.triu(h_r, 1)
        for k, hh, oo in zip(ks, hk, ok):
            ph = complex(np.exp(2j * np.pi * float(np.dot(k, R))))
            hh += h_r * ph + h_r.T * ph.conjugate()
            oo += o_r * ph + o_r.T * ph.conjugate()
    hd = (torch.rand(n, dtype=torch.float64, device=dev, generator=gen) * 1.5 - 1.0).to(torch.complex128)
    for hh in hk:
        hh.diagonal().copy_(hd)
    return hk, [_overlap(oo) for oo in ok]


def _sizes(case):
    """Uneven sizes: the ends of the range always, the rest log-uniform between them."""
    rng = np.random.default_rng(case["draws"])
    x = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["nprob"]))
    return [case["lo"], case["hi"]] + [int(round(v)) for v in x[2:]]


def _states(n, kt, full=False, gap=False):
    """(electrons, states): about a quarter electron per function (two states per atom with a
    gap); smearing takes n/8 states more."""
    nel = 4.0 * -(-n // 15) if gap else float(max(2, n // 4 // 2 * 2))
    k = int(nel // 2) + (n // 8 if kt > 0.0 else 0)
    return (float(n // 2), n) if full else (nel, max(1, min(n, k)))


def _gap(case):
    return case["geom"] == "cluster" and case["kt"] == 0.0


def _handle(n, k, nel, case, kt):
    h = egb.Handle(n, k, nel)
    h.use_current_stream()
    h.set_precision(egb.PREC_FP64 if case["prec"] == "f64" else egb.PREC_FP32_REFINE)
    if kt > 0.0:
        h.set_broadening(egb.OCC_FERMI, kt)
    return h


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "dm":
        n = case["n"]
        nel, k = _states(n, case["kt"], case["full"], _gap(case))
        st["H"], st["S"], _ = _real_problem(n, seed, case["geom"], gap=_gap(case))
        st["handle"] = _handle(n, k, nel, case, case["kt"])
    elif kind == "kpoints":
        n = case["n"]
        nel, k = _states(n, KT)
        st["H"], st["S"] = _kpoint_problems(n, case["nprob"], seed)
        st["k"], st["nel"] = [k] * case["nprob"], nel
        st["w"] = [1.0 / case["nprob"]] * case["nprob"]
        st["handle"] = _batch_handle(n, k, nel, case)
    elif kind == "mixed":
        ns = _sizes(case)
        probs = [_real_problem(n, seed * 64 + i, "cluster") for i, n in enumerate(ns)]
        st["H"], st["S"] = [p[0] for p in probs], [p[1] for p in probs]
        st["nel"], st["k"] = [list(x) for x in zip(*[_states(n, KT) for n in ns])]
        st["handle"] = _batch_handle(max(ns), max(st["k"]), st["nel"][0], case)
    elif kind == "fgrad":
        n = case["n"]
        nel, k = _states(n, KT)
        h, s, _ = _real_problem(n, seed, "cluster")
        st["H"], st["S"] = h.requires_grad_(True), s.requires_grad_(True)
        st["handle"] = _handle(n, k, nel, case, KT)
    elif kind == "egrad":
        n = case["n"]
        h, s, _ = _real_problem(n, seed, "cluster")
        st["H"], st["S"] = h.requires_grad_(True), s.requires_grad_(True)
        st["k"] = max(1, n // 8)
        st["w"], st["G"] = _egrad_loss(n, seed)
        st["handle"] = _handle(n, n, 0.0, case, 0.0)
    elif kind == "csc":
        n = case["n"]
        nel, k = _states(n, KT)
        h, s, mask = _real_problem(n, seed, "chain", CUTOFF)
        col, row = mask.nonzero(as_tuple=True)  # symmetric pattern: column by column
        ptr = torch.zeros(n + 1, dtype=torch.int64, device=h.device)
        ptr[1:] = torch.cumsum(mask.sum(1), 0)
        st["H"], st["S"] = h[col, row].contiguous(), s[col, row].contiguous()
        st["handle"] = _handle(n, k, nel, case, KT)
        st["handle"].set_csc(row.to(torch.int32).contiguous(), ptr.to(torch.int32))
    return st


def _batch_handle(n, k, nel, case):
    """The tuner's usual choice for these sizes, fixed: a program that cannot afford the
    tuning solves of a first call, and the same settings in every run."""
    h = _handle(n, k, nel, case, KT)
    h.set_batch_autotune(False)
    h.set_batch_streams(8)
    return h


def _egrad_loss(n, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed + 77)
    w = torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)
    g = torch.randn((n, n), dtype=torch.float64, device="cuda", generator=gen)
    return w, (g + g.T) * (0.5 / n)


# ---------------------------------------------------------------- one pass
def run(state):
    kind, h = state["kind"], state["handle"]
    if kind == "dm":
        p, e = h.dm_real(state["H"], state["S"])
        return {"P": p, "W": h.get_edm(), "energy": e, "mu": h.get_mu()}
    if kind == "kpoints":
        p, w, e, mu = h.dm_batched(state["H"], state["S"], state["k"], state["nel"],
                                   weights=state["w"], shared_mu=True)
        return {"P": p, "W": w, "energy": e, "mu": mu}
    if kind == "mixed":
        p, w, e, mu = h.dm_batched(state["H"], state["S"], state["k"], state["nel"], shared_mu=False)
        return {"P": p, "W": w, "energy": e, "mu": mu}
    if kind == "fgrad":
        f = ega.free_energy(state["H"], state["S"], h)
        gh, gs = torch.autograd.grad(f, (state["H"], state["S"]))
        return {"F": f.detach(), "gH": gh, "gS": gs}
    if kind == "egrad":
        ev, c = ega.eigh(state["H"], state["S"], h, state["k"])
        loss = (state["w"] * ev).sum() + ((state["G"] @ c) * c).sum()
        gh, gs = torch.autograd.grad(loss, (state["H"], state["S"]))
        return {"eval": ev.detach(), "loss": loss.detach(), "gH": gh, "gS": gs}
    p, e = h.dm_real_sparse(state["H"], state["S"])
    return {"P": p, "W": h.get_edm_sparse(), "energy": e}


# ---------------------------------------------------------------- work and reference
def work(case):
    kind = case["kind"]
    if kind == "mixed":
        ns = _sizes(case)
        one = [_work(n, _states(n, KT)[1]) for n in ns]
        return {"bytes": sum(b for b, _ in one), "flops": sum(f for _, f in one)}
    n = case["n"]
    if kind == "kpoints":
        b, f = _work(n, _states(n, KT)[1])
        return {"bytes": 2.0 * b * case["nprob"], "flops": 4.0 * f * case["nprob"]}
    if kind == "egrad":
        b, f = _work(n, n)
        return {"bytes": b + 8.0 * n, "flops": f + 4.0 * n ** 3}
    if kind == "csc":
        nnz = float(n) * min(n, 8 * 13)
        return {"bytes": 4.0 * 8.0 * nnz, "flops": _work(n, _states(n, KT)[1])[1]}
    k = _states(n, KT)[1]
    if kind == "dm":
        k = _states(n, case["kt"], case["full"], _gap(case))[1]
    b, f = _work(n, k)
    return {"bytes": b, "flops": f}


def _work(n, k):
    """H, S in and P, W out; Cholesky n^3/3, standard form n^3, tridiagonalisation 4n^3/3, the
    back-transformations of k vectors 5 n^2 k, P and W 2 n^2 k."""
    return 4.0 * 8.0 * n * n, 8.0 / 3.0 * n ** 3 + 7.0 * n * n * k


def _fermi(ev, wt, nel, kt):
    lo, hi = float(ev.min()) - 1.0, float(ev.max()) + 1.0

    def occ(m):
        return 2.0 / (1.0 + np.exp(np.clip((ev - m) / kt, -700.0, 700.0)))

    for _ in range(200):
        mid = 0.5 * (lo + hi)
        if float((wt * occ(mid)).sum()) > nel:
            hi = mid
        else:
            lo = mid
    mu = 0.5 * (lo + hi)
    return occ(mu), mu


def _eig(h, s):
    c = torch.linalg.cholesky(s)
    a = torch.linalg.solve_triangular(c, h, upper=False)
    a = torch.linalg.solve_triangular(c, a.mH, upper=False)
    ev, v = torch.linalg.eigh(0.5 * (a + a.mH))
    return ev, torch.linalg.solve_triangular(c.mH, v, upper=True)


def _pw(c, f, ev):
    f, ev = f.to(c.dtype), ev.to(c.dtype)
    return (c * f) @ c.mH, (c * (f * ev)) @ c.mH


def _dense_dm(h, s, nel, k, kt):
    ev, c = _eig(h, s)
    ev, c = ev[:k], c[:, :k]
    if kt > 0.0:
        f, mu = _fermi(ev.cpu().numpy(), np.ones(k), nel, kt)
        f = torch.from_numpy(f).to(ev.device)
    else:
        f = (nel - 2.0 * torch.arange(k, dtype=torch.float64, device=ev.device)).clamp(0.0, 2.0)
        mu = float(ev[int(math.ceil(nel / 2.0)) - 1])
    p, w = _pw(c, f, ev)
    return p, w, float((f * ev).sum()), mu, f


def exact(case, seed):
    kind = case["kind"]
    if kind == "mixed":
        ns = _sizes(case)
        out = [_dense_dm(*_real_problem(n, seed * 64 + i, "cluster")[:2], *_states(n, KT), KT)
               for i, n in enumerate(ns)]
        return {"P": [o[0] for o in out], "W": [o[1] for o in out], "energy": [o[2] for o in out],
                "mu": [o[3] for o in out]}
    n = case["n"]
    if n > EXACT_MAX:
        return None
    if kind == "dm":
        nel, k = _states(n, case["kt"], case["full"], _gap(case))
        p, w, e, mu, _ = _dense_dm(*_real_problem(n, seed, case["geom"], gap=_gap(case))[:2], nel, k, case["kt"])
        return {"P": p, "W": w, "energy": e, "mu": mu}
    if kind == "kpoints":
        nel, k = _states(n, KT)
        hk, sk = _kpoint_problems(n, case["nprob"], seed)
        eig = [_eig(h, s) for h, s in zip(hk, sk)]
        ev = np.concatenate([e[:k].cpu().numpy() for e, _ in eig])
        f, mu = _fermi(ev, np.full(ev.size, 1.0 / case["nprob"]), nel, KT)
        out = {"P": [], "W": [], "energy": [], "mu": mu}
        for i, (e, c) in enumerate(eig):
            fi = torch.from_numpy(f[i * k:(i + 1) * k]).to(e.device)
            p, w = _pw(c[:, :k], fi, e[:k])
            out["P"].append(p)
            out["W"].append(w)
            out["energy"].append(float((fi * e[:k]).sum()))
        return out
    if kind == "fgrad":
        nel, k = _states(n, KT)
        p, w, e, mu, f = _dense_dm(*_real_problem(n, seed, "cluster")[:2], nel, k, KT)
        x = (0.5 * f).clamp(1e-300, 1.0 - 1e-16)
        ent = float((2.0 * (x * x.log() + (1.0 - x) * torch.log1p(-x))).sum())
        return {"F": torch.tensor(e + KT * ent, dtype=torch.float64), "gH": p, "gS": -w}
    if kind == "egrad":
        h, s, _ = _real_problem(n, seed, "cluster")
        w, g = _egrad_loss(n, seed)
        k = max(1, n // 8)
        ev, c = _eig(h, s)
        o, v = c[:, :k], c[:, k:]
        m = 2.0 * (v.T @ g @ o) / (ev[None, :k] - ev[k:, None])
        ah, as_ = v @ m @ o.T, v @ (m * ev[:k]) @ o.T
        gh = (c * w) @ c.T + 0.5 * (ah + ah.T)
        gs = -(c * (w * ev)) @ c.T - 0.5 * (as_ + as_.T) - o @ (o.T @ g @ o) @ o.T
        return {"eval": ev, "loss": (w * ev).sum() + ((g @ o) * o).sum(), "gH": gh, "gS": gs}
    nel, k = _states(n, KT)
    h, s, mask = _real_problem(n, seed, "chain", CUTOFF)
    p, w, e, mu, _ = _dense_dm(h, s, nel, k, KT)
    col, row = mask.nonzero(as_tuple=True)
    return {"P": p[col, row], "W": w[col, row], "energy": e}
