"""What a user of the library has it compute, as cases that can be timed.

A case names a molecule of the repository's own workloads (a C_nH_{n+2}
zigzag chain or a hexagonal graphene flake with the even-tempered basis and
the minimal ris auxiliary sets), the precision and the response problem, and
one call of the public interface: the response operator on a block of
vectors, a new geometry's integrals and B tensors, gradients, derivative
couplings, the Z-vector solve, a whole evaluation, or one step of a
surface-hopping trajectory.  Molecular orbitals, orbital energies and
amplitudes are drawn from the seed as the workloads draw them (Haar-random
rotations of an orthonormal set, uniform energies).

`exact` evaluates the same quantities from their formulas in 64 bits with
torch: McMurchie-Davidson integrals, the literal resolution of the identity
with M^-1 by a linear solve, dense diagonalisation where it is small enough,
and gradients by reverse-mode differentiation of the pair energies.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2511_18233_gb300 import ris, synth

CX = 0.25            # fraction of exact exchange of every case (the library's default)
SIGMA = 0.05         # thermal displacement of a trajectory step, Angstrom
LINDEP = synth.SERVING_LINDEP
DEV = "cuda"


# ------------------------------------------------------------------ the cases

def _case(kind, mol, size, precision="f64", rpa=False, count=1):
    return {"kind": kind, "mol": mol, "size": size, "precision": precision, "rpa": rpa,
            "count": count}


def listed():
    """kind / what `count` counts: apply: vectors; geometry: probe vectors; grad: states;
    nac: adjacent pairs; zvector: right-hand sides; eval, step: states."""
    rows = [
        # the smallest call: one operator product of the 10-atom chain (launches and latency)
        ("apply_f64_c4h6", _case("apply", "chain", 4, count=1)),
        # a Davidson block of the 42-atom chain: correction vectors of 10 states
        ("apply_f64_c20h22", _case("apply", "chain", 20, count=10)),
        # the first block of a mixed-precision Davidson for 10 states (10 + 8 vectors)
        ("apply_mixed_c20h22", _case("apply", "chain", 20, "mixed", count=18)),
        # full-RPA products (A+B)X, (A-B)X on the largest flake, a few unconverged states
        ("apply_rpa_f64_c54h18", _case("apply", "flake", 7.0, rpa=True, count=4)),
        # a new geometry in FP64: integrals, metric factors, B tensors, one product
        ("geometry_f64_c20h22", _case("geometry", "chain", 20, count=1)),
        # gradients of all ten states in FP64 at given amplitudes
        ("grad_f64_c20h22", _case("grad", "chain", 20, count=10)),
        # couplings between the adjacent states in mixed precision at given amplitudes
        ("nac_mixed_c20h22", _case("nac", "chain", 20, "mixed", count=9)),
        # the backward of the differentiable RPA energy: one state's gradient on a flake
        ("grad_rpa_f64_c24h12", _case("grad", "flake", 5.0, rpa=True, count=1)),
        # the ris Z-vector solve behind a relaxed gradient
        ("zvector_f64_c12h14", _case("zvector", "chain", 12, count=3)),
        # a whole FP64 evaluation of the small chain through host arrays: 5 states,
        # 5 gradients, the 1-2 coupling
        ("eval_f64_c4h6", _case("eval", "chain", 4, count=5)),
        # the headline evaluation: 10 states, 10 gradients, 9 couplings, mixed precision
        ("eval_mixed_c20h22", _case("eval", "chain", 20, "mixed", count=10)),
        # one served surface-hopping step: new geometry, Davidson seeded with the last
        # step's amplitudes, phases, active-state gradient, couplings, T_IJ
        ("step_mixed_c24h12", _case("step", "flake", 5.0, "mixed", count=7)),
    ]
    return [dict(c, name=n) for n, c in rows]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo - 0.49), math.log(hi + 0.49)))))))


def draw(rng):
    """Another case of the same ranges: chains C2 .. C40, flakes of 4 .. 7 Angstrom, blocks of
    1 .. 18 vectors, 1 .. 10 states, at most the cost of the largest listed case."""
    top = max(_seconds(c) for c in listed())
    while True:
        kind = rng.choice(["apply", "apply", "geometry", "grad", "nac", "zvector", "eval", "step"])
        mixed = kind == "step" or (kind != "zvector" and rng.random() < 0.4)
        rpa = kind in ("apply", "grad") and not mixed and rng.random() < 0.35
        count = _log_int(rng, 1, 18 if kind == "apply" else 10)
        if kind == "eval" and not mixed:
            mol, size, count = "chain", _log_int(rng, 2, 6), min(count, 6)
        elif rng.random() < 0.65:
            mol, size = "chain", _log_int(rng, 2, 40)
        else:
            mol, size = "flake", _valid_radius(round(rng.uniform(4.0, 7.0), 2))
        if kind in ("eval", "step"):
            count = max(count, 3)
        if kind == "eval" and mol == "flake":
            continue  # flakes are evaluated step by step along trajectories
        c = _case(kind, mol, size, "mixed" if mixed else "f64", rpa, count)
        if _seconds(c) <= top:
            return c


def _valid_radius(r):
    while True:
        try:
            synth.flake_geometry(r)
            return r
        except ValueError:
            r = round(r - 0.01, 2)


# ------------------------------------------------------------------ molecules

@functools.lru_cache(maxsize=None)
def _molecule(mol, size):
    """Geometry, shells and occupation of a molecule (no MOs)."""
    el, xyz = synth.chain_geometry(int(size)) if mol == "chain" else synth.flake_geometry(float(size))
    return synth.make_molecule(mol, el, xyz, 0, not (mol == "chain" and size <= 4), with_mo=False)


def _functions(shells):
    """Per cartesian function: atom, (lx, ly, lz), exponent, normalisation."""
    at, cart, ex = [], [], []
    for s in shells:
        for c in synth.cart_components(int(s["l"])):
            at.append(int(s["atom"]))
            cart.append(c)
            ex.append(float(s["exp"]))
    cart, ex = np.array(cart), np.array(ex)
    df = np.array([1.0, 1.0, 3.0])  # (2l-1)!!
    norm = (2 * ex / np.pi) ** 0.75 * (4 * ex) ** (cart.sum(1) / 2) / np.sqrt(df[cart].prod(1))
    return np.array(at), cart, ex, norm


@functools.lru_cache(maxsize=8)
def _orthonormal(mol, size, cutoff):
    """S^-1/2 (cutoff 0) or U lambda^-1/2 over the overlap eigenvalues above the cutoff."""
    m = _molecule(mol, size)
    at, cart, ex, norm = _functions(m.shells)
    p = ex[:, None] + ex[None, :]
    S = np.outer(norm, norm)
    for d in range(3):
        A = m.coords[at, d]
        PA = -ex[None, :] / p * (A[:, None] - A[None, :])
        PB = ex[:, None] / p * (A[:, None] - A[None, :])
        s = {(0, 0): np.exp(-ex[:, None] * ex[None, :] / p * (A[:, None] - A[None, :]) ** 2)
             * np.sqrt(np.pi / p)}
        zero = np.zeros_like(p)
        for i in range(3):
            for j in range(3):
                if (i, j) == (0, 0):
                    continue
                if i > 0:
                    r, x, a, b = (i - 1, j), PA, (i - 2, j), (i - 1, j - 1)
                else:
                    r, x, a, b = (i, j - 1), PB, (i - 1, j - 1), (i, j - 2)
                s[i, j] = x * s[r] + (max(r[0], 0) * s.get(a, zero) + max(r[1], 0) * s.get(b, zero)) / (2 * p)
        li, lj = np.broadcast_arrays(cart[:, d][:, None], cart[:, d][None, :])
        S *= np.choose(3 * li + lj, [s[i, j] for i in range(3) for j in range(3)])
    w, U = np.linalg.eigh(0.5 * (S + S.T))
    if cutoff:
        return U[:, w > cutoff] * w[w > cutoff] ** -0.5
    return (U * w ** -0.5) @ U.T


def _dims(case):
    m = _molecule(case["mol"], case["size"])
    n, o = m.nao, m.nocc
    nmo = _orthonormal(case["mol"], case["size"], LINDEP).shape[1] if _moving(case) else n
    return n, o, nmo - o, m.naux("J"), m.naux("K")


def _moving(case):
    """Cases whose geometry moves while the MOs stay: serving MOs, thermal displacements."""
    return case["kind"] in ("geometry", "step")


# ------------------------------------------------------------------ inputs

def _inputs(case, seed):
    """Everything a program has in hand, as numpy arrays."""
    m = _molecule(case["mol"], case["size"])
    rng = np.random.default_rng([2511, seed])
    base = _orthonormal(case["mol"], case["size"], LINDEP if _moving(case) else 0.0)
    C = np.ascontiguousarray(base @ synth.haar_orthogonal(base.shape[1], rng))
    o, v = m.nocc, C.shape[1] - m.nocc
    eps = synth.orbital_energies(o, v, rng)
    ref = m.coords
    coords = synth.perturb(ref, SIGMA, rng) if _moving(case) else ref.copy()
    count = case["count"]
    nst = count + 1 if case["kind"] == "nac" else count
    gap = eps[o:][None, :] - eps[:o][:, None]
    x = rng.standard_normal((nst, o, v))
    y = None
    if case["kind"] in ("grad", "nac"):
        # amplitudes like a converged state's: large on the small orbital-energy differences
        w = np.sort(rng.uniform(0.6, 0.95, nst)) * gap.min()
        x /= gap[None] - w[:, None, None]
        x = np.linalg.qr(x.reshape(nst, -1).T)[0].T.reshape(nst, o, v)
        if case["rpa"]:
            y = 0.05 * rng.standard_normal(x.shape) / (gap[None] + w[:, None, None])
            y *= 0.1 / np.linalg.norm(y.reshape(nst, -1), axis=1)[:, None, None]
            x *= math.sqrt(1.01)
    else:
        w = gap.min() + 0.02 * np.arange(nst)
        x = np.linalg.qr((x / np.sqrt(gap)[None]).reshape(nst, -1).T)[0].T.reshape(nst, o, v)
    velocity = rng.normal(size=(m.natm, 3)) * 1e-4
    c = np.ascontiguousarray
    return m, ref, coords, C, eps, c(x), None if y is None else c(y), c(w), velocity


def prepare(case, seed):
    m, ref, coords, C, eps, x, y, w, velocity = _inputs(case, seed)
    dev = lambda a: None if a is None else torch.as_tensor(a, dtype=torch.float64, device=DEV)  # noqa: E731
    mixed = case["precision"] == "mixed"
    ctx = ris.Context(precision=ris.MIXED if mixed else ris.FP64, rpa=int(case["rpa"]), cx=CX)
    shells = tuple(ris._shells(a) for a in (m.shells, m.aux_j, m.aux_k))
    n, o, v = m.nao, m.nocc, C.shape[1] - m.nocc
    kind, count = case["kind"], case["count"]
    s = {"kind": kind, "rpa": case["rpa"], "ctx": ctx, "shells": shells, "nocc": o, "count": count,
         "coords": coords, "C": dev(C), "eps": dev(eps)}
    new = lambda *shape: torch.zeros(shape, dtype=torch.float64, device=DEV)  # noqa: E731
    if kind == "eval" and n <= 250:  # small molecules: a program with host arrays
        s.update(C=C, eps=eps, host=True)
    elif kind == "eval":
        s.update(host=False, omega=new(count), X=new(count, o, v), grad=new(count, m.natm, 3),
                 nac=new(max(count - 1, 1), m.natm, 3))
    if kind in ("apply", "grad", "nac", "zvector"):  # the context holds this geometry
        ctx.build_aux(coords, *shells)
        ctx.build_B(s["C"], s["eps"], o)
    if kind in ("apply", "geometry"):
        s.update(X=dev(x), out=new(count, o, v), out2=new(count, o, v) if case["rpa"] else None)
    elif kind == "zvector":
        s.update(rhs=dev(x), Z=new(count, o, v))
    elif kind in ("grad", "nac"):
        s.update(X=dev(x), Y=dev(y), omega=w, out=new(count, m.natm, 3),
                 pairs=[(k, k + 1) for k in range(count)])
    elif kind == "step":
        # the trajectory's previous step: its amplitudes stay on the device
        active = count // 2
        s.update(X0=new(count, o, v), X=new(count, o, v), omega=new(count), active=active,
                 pairs=[(active - 1, active), (active, active + 1)] if active else [(0, 1)],
                 velocity=velocity)
        ctx.build_aux(ref, *shells)
        ctx.build_B(s["C"], s["eps"], o)
        ctx.excite(count, out=(s["omega"], s["X0"], None))
    return s


def run(s):
    ctx, kind, count = s["ctx"], s["kind"], s["count"]
    if kind == "apply":
        r = ctx.apply(s["X"], out=s["out"], out2=s["out2"])
        return {"AX": r} if not s["rpa"] else {"P": r[0], "M": r[1]}
    if kind == "grad":
        return {"grad": ctx.gradient(range(count), X=s["X"], Y=s["Y"], out=s["out"])}
    if kind == "nac":
        return {"nac": ctx.nac(s["pairs"], X=s["X"], omega=s["omega"], out=s["out"])}
    if kind == "zvector":
        return {"Z": ctx.zvector(s["rhs"], out=s["Z"])}
    ctx.build_aux(s["coords"], *s["shells"])
    ctx.build_B(s["C"], s["eps"], s["nocc"])
    if kind == "geometry":
        return {"AX": ctx.apply(s["X"], out=s["out"])}
    if kind == "eval":
        adjacent = [(k, k + 1) for k in range(1 if s["host"] else count - 1)]
        if s["host"]:
            om, X = ctx.excite(count)
            return {"omega": om, "X": X, "grad": ctx.gradient(range(count)), "nac": ctx.nac(adjacent)}
        om, X = ctx.excite(count, out=(s["omega"], s["X"], None))
        return {"omega": om, "X": X, "grad": ctx.gradient(range(count), out=s["grad"]),
                "nac": ctx.nac(adjacent, out=s["nac"])}
    om, X = ctx.excite_guess(count, s["X0"], out=(s["omega"], s["X"], None))
    signs = ctx.phase_align(s["X0"], X_out=X)
    grad = ctx.gradient([s["active"]])
    nac = ctx.nac(s["pairs"])
    return {"omega": om, "X": X, "signs": signs, "grad": grad, "nac": nac,
            "T": ctx.time_coupling(nac, s["velocity"])}


# ------------------------------------------------------------------ work

def work(case):
    """The contractions of the method (integral recursions not counted) and the tensors that
    a pass has to read or write: B tensors, derivative integrals, inputs and results."""
    n, o, v, nJ, nK = _dims(case)
    nov, count, rpa = o * v, case["count"], case["rpa"]
    prod = 4.0 * nov * nJ + 2.0 * o * o * v * nK + 2.0 * o * v * v * nK
    held = 8.0 * (nov * nJ + o * o * nK + v * v * nK)
    if rpa or case["kind"] == "zvector":
        prod += 4.0 * o * o * v * nK
        held += 8.0 * nov * nK
    build = (2.0 * o * n * n * nJ + 2.0 * nov * n * nJ + 2.0 * nov * nJ * nJ + 2.0 * v * n * n * nK
             + 2.0 * v * v * n * nK + 2.0 * v * v * nK * nK + 2.0 * o * o * n * nK)
    d = 4.0 if case["precision"] == "mixed" else 8.0
    pair = (2 if rpa else 1) * (2.0 * o * v * v * nK + 2.0 * o * o * v * nK + 4.0 * n * o * o * nK
                                + 4.0 * n * n * o * nK) + 6.0 * n * n * nK
    state = 6.0 * n * n * nJ + 2.0 * n * nov + 2.0 * n * n * v
    ints = d * 3.0 * n * n * max(nJ, nK)
    kind = case["kind"]
    if kind == "apply":
        return {"bytes": held + (24.0 if rpa else 16.0) * nov * count, "flops": prod * count}
    if kind == "geometry":
        return {"bytes": held + 8.0 * n * (o + v) + 16.0 * nov * count, "flops": build + prod * count}
    if kind in ("grad", "nac"):
        states = count + (kind == "nac")
        return {"bytes": held + ints + 8.0 * nov * states, "flops": pair * count + state * states}
    if kind == "zvector":
        return {"bytes": held + 16.0 * nov * count, "flops": 10.0 * prod * count}
    pairs = count + (count - 1 if kind == "eval" else 0) if kind == "eval" else 3
    return {"bytes": held + ints + 8.0 * n * (o + v) + 8.0 * nov * count,
            "flops": build + 6.0 * count * prod + pairs * pair + count * state}


def _seconds(case):
    """Rough duration of a pass, to keep drawn cases within the listed ones."""
    w = work(case)
    return w["flops"] / (4e13 if case["precision"] == "mixed" else 1e12) + w["bytes"] / 2e12 + 1e-4


# ------------------------------------------------------------------ 64-bit values

def exact(case, seed):
    kind, count = case["kind"], case["count"]
    n, o, v, nJ, nK = _dims(case)
    if kind in ("eval", "step") and o * v > 3000:
        return None  # a dense diagonalisation would take too long
    if kind in ("grad", "nac") and n * n * (nJ + 5.0 * nK) * count > 2.5e9:
        return None
    m, ref, coords, C, eps, x, y, w, velocity = _inputs(case, seed)
    sets = [(a, _Integrals(m, a)) for a in (m.aux_j, m.aux_k)]
    t = lambda a: None if a is None else torch.as_tensor(a, dtype=torch.float64, device=_device())  # noqa: E731
    R, Ct, X, Y = t(coords), t(C), t(x), t(y)
    with torch.no_grad():
        TJ, TK = (i.three_centre(R) for _, i in sets)
        MJ, MK = (i.metric(R) for _, i in sets)
        op = _Operator(TJ, MJ, TK, MK, Ct, t(eps), o)
        if kind in ("apply", "geometry"):
            P, M = op.products(X, case["rpa"])
            return {"P": P, "M": M} if case["rpa"] else {"AX": P}
        if kind == "zvector":
            return {"Z": op.solve(X)}
        out = {}
        if kind in ("eval", "step"):
            om, X = op.lowest(count)
            w = om.cpu().numpy()
            if kind == "step":
                out["signs"] = None
                X0 = _previous_step(m, sets, t(ref), Ct, t(eps), o, count)
                X = X * _signs(X, X0)[:, None, None]
            out.update(omega=om, X=X)
    active = count // 2
    near = [(active - 1, active), (active, active + 1)] if active else [(0, 1)]
    gpairs = {"grad": range(count), "eval": range(count), "step": [active]}.get(kind, [])
    npairs = {"nac": [(k, k + 1) for k in range(count)], "step": near,
              "eval": [(k, k + 1) for k in range(1 if n <= 250 else count - 1)]}.get(kind, [])
    pairs = [(k, k) for k in gpairs] + npairs
    g = _pair_gradients(sets, R, Ct, o, X, Y, pairs, (TJ, MJ, TK, MK))
    if len(gpairs):
        out["grad"] = g[: len(gpairs)]
    if npairs:
        den = torch.as_tensor([w[j] - w[i] for i, j in npairs], dtype=torch.float64, device=g.device)
        out["nac"] = g[len(gpairs):] / den[:, None, None]
    if kind == "step":
        out["T"] = (out["nac"] * t(velocity)[None]).sum((1, 2))
    return out


def _device():
    return DEV if torch.cuda.is_available() else "cpu"


def _previous_step(m, sets, R, C, eps, o, count):
    T = [i.three_centre(R) for _, i in sets]
    M = [i.metric(R) for _, i in sets]
    return _Operator(T[0], M[0], T[1], M[1], C, eps, o).lowest(count)[1]


def _signs(X, X0):
    """Sign of the overlap over the five largest determinants of the previous step."""
    a, b = X.reshape(len(X), -1), X0.reshape(len(X0), -1)
    top = b.abs().topk(5, dim=1).indices
    s = (a.gather(1, top) * b.gather(1, top)).sum(1)
    return torch.where(s < 0, -1.0, 1.0).to(X.dtype)


class _Operator:
    """A (and B) of the ris problem from the three-centre integrals and the metrics."""

    def __init__(self, TJ, MJ, TK, MK, C, eps, o):
        self.o, Co, Cv = o, C[:, :o], C[:, o:]
        mo = lambda T, l, r: torch.einsum("mia,mp->pia", torch.einsum("mnP,na->mPa", T, r), l)  # noqa: E731
        self.ovJ = mo(TJ, Co, Cv)            # [i][P][a]
        self.oo, self.ov, self.vv = mo(TK, Co, Co), mo(TK, Co, Cv), mo(TK, Cv, Cv)
        self.MJ, self.MK = MJ, MK
        sol = lambda t: torch.linalg.solve(MK, t.permute(1, 0, 2).reshape(t.shape[1], -1)).reshape(  # noqa: E731
            t.shape[1], t.shape[0], t.shape[2]).permute(1, 0, 2)
        self.moo, self.mov = sol(self.oo), sol(self.ov)
        self.de = eps[o:][None, :] - eps[:o][:, None]

    def parts(self, X):
        u = torch.einsum("iPa,ia->P", self.ovJ, X)
        J = torch.einsum("iPa,P->ia", self.ovJ, torch.linalg.solve(self.MJ, u))
        K1 = torch.einsum("jPa,aPb->jb", torch.einsum("iPj,ja->iPa", self.moo, X), self.vv)
        K2 = torch.einsum("iPj,jPa->ia", torch.einsum("iPb,jb->iPj", self.mov, X), self.ov)
        return J, K1, K2

    def products(self, X, rpa):
        P, M = [], []
        for x in X:
            J, K1, K2 = self.parts(x)
            P.append(self.de * x + (4 * J - CX * (K1 + K2) if rpa else 2 * J - CX * K1))
            M.append(self.de * x - CX * (K1 - K2))
        return torch.stack(P), torch.stack(M)

    def solve(self, rhs):
        """(A+B) Z = rhs by conjugate gradients with the Coulomb-exact preconditioner."""
        o, v = self.de.shape
        B = self.ovJ.permute(0, 2, 1).reshape(o * v, -1)
        L = torch.linalg.cholesky(self.MJ)
        B = torch.linalg.solve_triangular(L, B.T, upper=False).T
        d = self.de.reshape(-1)
        cap = torch.eye(B.shape[1], dtype=B.dtype, device=B.device) + 4 * (B.T / d) @ B
        def pre(r):
            q = r / d[None]
            return q - 4 * (torch.linalg.solve(cap, B.T @ q.T).T @ B.T) / d[None]
        b = rhs.reshape(len(rhs), -1)
        z = torch.zeros_like(b)
        r = b.clone()
        p = q = pre(r)
        rq = (r * q).sum(1)
        for _ in range(60):
            ap = self.products(p.reshape(rhs.shape), True)[0].reshape(b.shape)
            a = rq / (p * ap).sum(1)
            z, r = z + a[:, None] * p, r - a[:, None] * ap
            if bool((r.norm(dim=1) <= 1e-14 * b.norm(dim=1)).all()):
                break
            q = pre(r)
            new = (r * q).sum(1)
            p, rq = q + (new / rq)[:, None] * p, new
        return z.reshape(rhs.shape)

    def lowest(self, count):
        o, v = self.de.shape
        B = self.ovJ.permute(1, 0, 2).reshape(-1, o * v)
        A = 2 * B.T @ torch.linalg.solve(self.MJ, B)
        A -= CX * torch.einsum("iPj,aPb->iajb", self.moo, self.vv).reshape(o * v, o * v)
        A = 0.5 * (A + A.T) + torch.diag(self.de.reshape(-1))
        w, V = torch.linalg.eigh(A)
        V = V[:, :count].T
        top = V.abs().argmax(1, keepdim=True)
        V = V * torch.sign(V.gather(1, top))
        return w[:count], V.reshape(count, o, v)


def _pair_energy(X, Y, I, J, T, C, o):
    """E_IJ = 1/2 [R_I (A+B) R_J + L_I (A-B) L_J] without the orbital energies."""
    TJ, MJ, TK, MK = T
    Co, Cv = C[:, :o], C[:, o:]
    R = lambda k: X[k] if Y is None else X[k] + Y[k]  # noqa: E731
    L = lambda k: X[k] if Y is None else X[k] - Y[k]  # noqa: E731
    D = lambda A: Co @ A @ Cv.T  # noqa: E731
    u = [torch.einsum("mnP,mn->P", TJ, D(R(k))) for k in (I, J)]
    E = 2 * u[0] @ torch.linalg.solve(MJ, u[1])
    half = torch.einsum("mnP,ni->mPi", TK, Co)
    oo = torch.einsum("mPi,mj->jPi", half, Co)
    moo = torch.linalg.solve(MK, oo.permute(1, 0, 2).reshape(oo.shape[1], -1)).reshape(-1, o, o)
    for f, U, V in ((0.5, R(I), R(J)), (0.5, L(I), L(J))) if Y is not None else ((1.0, R(I), R(J)),):
        # sum (ij|ab) U_ia V_jb with the virtual indices folded into the AO ones
        QU, QV = U @ Cv.T, V @ Cv.T
        g = torch.einsum("iPm,jm->ijP", torch.einsum("mnP,in->iPm", TK, QU), QV)
        E = E - CX * f * torch.einsum("ijP,Pij->", g, moo)
    if Y is not None:
        ov = torch.einsum("mPi,ma->iPa", half, Cv)
        for f, U, V in ((-0.5, R(I), R(J)), (0.5, L(I), L(J))):
            e1 = torch.einsum("ia,jPa->Pij", U, ov)
            e2 = torch.einsum("jb,iPb->Pji", V, ov)
            sol = torch.linalg.solve(MK, e1.reshape(e1.shape[0], -1)).reshape(e1.shape)
            E = E + CX * f * torch.einsum("Pij,Pji->", sol, e2)
    return E


def _pair_gradients(sets, R, C, o, X, Y, pairs, T):
    dens = [[], [], [], []]
    for I, J in pairs:
        leaf = [t.detach().clone().requires_grad_(True) for t in T]
        g = torch.autograd.grad(_pair_energy(X, Y, I, J, leaf, C, o), leaf)
        for k in range(4):
            dens[k].append(g[k])
    out = torch.zeros((len(pairs),) + tuple(R.shape), dtype=R.dtype, device=R.device)
    for k, (_, ints) in enumerate(sets):
        out += ints.gradient(R, dens[2 * k], dens[2 * k + 1])
    return out


# ---------------------------------------------------------------- integrals

class _Boys(torch.autograd.Function):
    """F_0 .. F_n of T, stacked; dF_m/dT = -F_{m+1}."""

    @staticmethod
    def forward(ctx, T, n):
        big = T > 35.0
        t = torch.where(big, torch.zeros_like(T), T)
        top = torch.zeros_like(T)
        term = torch.full_like(T, 1.0 / (2 * n + 3))
        for k in range(160):  # F_{n+1} by its ascending series
            top = top + term
            term = term * (2 * t / (2 * n + 2 * k + 5))
        e = torch.exp(-t)
        F = [None] * (n + 2)
        F[n + 1] = e * top
        for m in range(n, -1, -1):
            F[m] = (2 * t * F[m + 1] + e) / (2 * m + 1)
        tb = torch.where(big, T, torch.ones_like(T))
        up, eb = 0.5 * torch.sqrt(math.pi / tb) * torch.erf(torch.sqrt(tb)), torch.exp(-tb)
        for m in range(n + 2):
            F[m] = torch.where(big, up, F[m])
            up = ((2 * m + 1) * up - eb) / (2 * tb)
        F = torch.stack(F)
        ctx.save_for_backward(F)
        return F[: n + 1]

    @staticmethod
    def backward(ctx, g):
        (F,) = ctx.saved_tensors
        return -(F[1:] * g).sum(0), None


def _hermite_R(n, alpha, X):
    """R_tuv for t + u + v <= n at the vectors X[..., 3], as {(t, u, v): tensor}."""
    F = _Boys.apply(alpha * (X * X).sum(-1), n)
    lev = {(0, 0, 0): [(-2 * alpha) ** m * F[m] for m in range(n + 1)]}
    for total in range(1, n + 1):
        for t in range(total, -1, -1):
            for u in range(total - t, -1, -1):
                tuv = (t, u, total - t - u)
                d = next(k for k in range(3) if tuv[k])
                one = tuple(c - (k == d) for k, c in enumerate(tuv))
                two = tuple(c - 2 * (k == d) for k, c in enumerate(tuv))
                f = tuv[d] - 1
                lev[tuv] = [X[..., d] * lev[one][m + 1] + (f * lev[two][m + 1] if f else 0.0)
                            for m in range(n - total + 1)]
    return {k: v[0] for k, v in lev.items()}


def _hermite_E(la, lb, a, b, A, B):
    """E[i][j][t] of one direction of a Gaussian pair."""
    p = a + b
    PA, PB = -b / p * (A - B), a / p * (A - B)
    E = {(0, 0, 0): torch.exp(-a * b / p * (A - B) ** 2)}
    get = lambda i, j, t: E.get((i, j, t), 0.0)  # noqa: E731
    for i in range(la + 1):
        for j in range(lb + 1):
            if i + j == 0:
                continue
            pi, pj, x = (i - 1, j, PA) if i else (i, j - 1, PB)
            for t in range(i + j + 1):
                E[i, j, t] = get(pi, pj, t - 1) / (2 * p) + x * get(pi, pj, t) + (t + 1) * get(pi, pj, t + 1)
    return E


class _Integrals:
    """(mu nu|P) and (P|Q) of one auxiliary set, and their derivatives contracted with densities."""

    def __init__(self, m, aux, chunk=3_000_000):
        self.ao, self.aux, self.natm, self.nao = _shell_groups(m.shells), _shell_groups(aux), m.natm, m.nao
        self.naux, self.chunk = sum(synth.ncart(int(s["l"])) for s in aux), chunk

    def _classes(self, dev):
        for la in self.ao:
            for lb in self.ao:
                if lb > la:
                    continue
                a, b = self.ao[la], self.ao[lb]
                ia, ib = np.meshgrid(np.arange(len(a["at"])), np.arange(len(b["at"])), indexing="ij")
                keep = (ia >= ib) if la == lb else np.ones_like(ia, bool)
                ia, ib = ia[keep], ib[keep]
                for lc in self.aux:
                    step = max(1, self.chunk // len(self.aux[lc]["at"]))
                    for s in range(0, len(ia), step):
                        yield la, lb, lc, ia[s:s + step], ib[s:s + step]

    def _block(self, R, la, lb, lc, ia, ib):
        """Integrals [component a][component b][component c][pair][aux shell]."""
        f = lambda x: torch.as_tensor(x, dtype=R.dtype, device=R.device)  # noqa: E731
        a, b, c = self.ao[la], self.ao[lb], self.aux[lc]
        ea, eb, ec = f(a["ex"][ia]), f(b["ex"][ib]), f(c["ex"])
        A, B, Cc = R[a["at"][ia]], R[b["at"][ib]], R[c["at"]]
        p = ea + eb
        P = (ea[:, None] * A + eb[:, None] * B) / p[:, None]
        alpha = p[:, None] * ec[None, :] / (p[:, None] + ec[None, :])
        Rt = _hermite_R(la + lb + lc, alpha, P[:, None, :] - Cc[None, :, :])
        pre = 2 * math.pi ** 2.5 / (p[:, None] * ec[None, :] * torch.sqrt(p[:, None] + ec[None, :]))
        E = [_hermite_E(la, lb, ea, eb, A[:, d], B[:, d]) for d in range(3)]
        tuv = [(t, u, l - t - u) for l in range(la + lb + 1) for t in range(l + 1) for u in range(l - t + 1)]
        ca, cb, cc = (synth.cart_components(l) for l in (la, lb, lc))
        zero = torch.zeros_like(p)
        H = torch.stack([torch.stack([
            E[0].get((x[0], y[0], k[0]), zero) * E[1].get((x[1], y[1], k[1]), zero)
            * E[2].get((x[2], y[2], k[2]), zero) * (_norm(x, a["ex"][ia], f) * _norm(y, b["ex"][ib], f))
            for k in tuv]) for x in ca for y in cb])
        out = []
        for z in cc:
            # auxiliary factor: 1 (s) or Lambda_1 / 2 gamma (p), with (-1)^tau for the ket
            g = pre * _norm(z, c["ex"], f)[None, :] * ((-0.5 / ec[None, :]) if lc else 1.0)
            G = torch.stack([Rt[tuple(k[d] + z[d] for d in range(3))] for k in tuv]) * g
            out.append(torch.einsum("ktp,tpc->kpc", H, G))
        v = torch.stack(out)  # [c comp][(a,b) comp][pair][aux]
        return v.reshape(len(cc), len(ca), len(cb), len(ia), len(c["at"]))

    def _where(self, la, lb, lc, ia, ib, dev):
        a, b, c = self.ao[la], self.ao[lb], self.aux[lc]
        t = lambda x: torch.as_tensor(x, device=dev)  # noqa: E731
        comp = lambda l: np.arange(synth.ncart(l))  # noqa: E731
        mu = (a["off"][ia][None, None, None, :, None] + comp(la)[None, :, None, None, None])
        nu = (b["off"][ib][None, None, None, :, None] + comp(lb)[None, None, :, None, None])
        P = (c["off"][None, None, None, None, :] + comp(lc)[:, None, None, None, None])
        return t(mu), t(nu), t(P)

    def three_centre(self, R):
        T = torch.zeros((self.nao, self.nao, self.naux), dtype=R.dtype, device=R.device)
        for la, lb, lc, ia, ib in self._classes(R.device):
            v = self._block(R, la, lb, lc, ia, ib)
            mu, nu, P = self._where(la, lb, lc, ia, ib, R.device)
            T[mu, nu, P] = v
            T[nu, mu, P] = v
        return T

    def metric(self, R):
        M = torch.zeros((self.naux, self.naux), dtype=R.dtype, device=R.device)
        f = lambda x: torch.as_tensor(x, dtype=R.dtype, device=R.device)  # noqa: E731
        rows = []
        for l1, s1 in self.aux.items():
            for l2, s2 in self.aux.items():
                g1, g2 = f(s1["ex"])[:, None], f(s2["ex"])[None, :]
                X = R[s1["at"]][:, None, :] - R[s2["at"]][None, :, :]
                Rt = _hermite_R(l1 + l2, g1 * g2 / (g1 + g2), X)
                pre = 2 * math.pi ** 2.5 / (g1 * g2 * torch.sqrt(g1 + g2))
                for i, x in enumerate(synth.cart_components(l1)):
                    for j, y in enumerate(synth.cart_components(l2)):
                        w = pre * _norm(x, s1["ex"], f)[:, None] * _norm(y, s2["ex"], f)[None, :]
                        w = w * (0.5 / g1 if l1 else 1.0) * (-0.5 / g2 if l2 else 1.0)
                        v = w * Rt[tuple(x[d] + y[d] for d in range(3))]
                        at = (torch.as_tensor(s1["off"] + i, device=R.device)[:, None],
                              torch.as_tensor(s2["off"] + j, device=R.device)[None, :])
                        rows.append((at, v))
        for at, v in rows:
            M = M.index_put(at, v)
        return M

    def gradient(self, R, dT, dM):
        """sum dT_{mn,P} d(mn|P)/dR + sum dM_PQ d(P|Q)/dR for lists of densities."""
        out = torch.zeros((len(dT),) + tuple(R.shape), dtype=R.dtype, device=R.device)
        for la, lb, lc, ia, ib in self._classes(R.device):
            mu, nu, P = self._where(la, lb, lc, ia, ib, R.device)
            r = R.detach().clone().requires_grad_(True)
            v = self._block(r, la, lb, lc, ia, ib)
            once = torch.where(mu == nu, 0.5, 1.0).to(R.dtype)
            if la == lb:  # the diagonal shell pairs hold both orders of their components
                once = torch.where(torch.as_tensor(ia == ib, device=R.device)[None, None, None, :, None],
                                   0.5, 1.0).to(R.dtype) * torch.ones_like(once)
            for k, D in enumerate(dT):
                out[k] += torch.autograd.grad(v, r, (D[mu, nu, P] + D[nu, mu, P]) * once,
                                              retain_graph=True)[0]
        r = R.detach().clone().requires_grad_(True)
        M = self.metric(r)
        for k, D in enumerate(dM):
            out[k] += torch.autograd.grad(M, r, D, retain_graph=True)[0]
        return out


def _norm(cart, ex, f):
    df = {0: 1.0, 1: 1.0, 2: 3.0}
    l = sum(cart)
    return f((2 * ex / np.pi) ** 0.75 * (4 * ex) ** (l / 2) / math.sqrt(math.prod(df[c] for c in cart)))


def _shell_groups(shells):
    """{l: atoms, exponents, first functions of the shells of that angular momentum}."""
    first, out = 0, {}
    for s in shells:
        g = out.setdefault(int(s["l"]), {"at": [], "ex": [], "off": []})
        g["at"].append(int(s["atom"]))
        g["ex"].append(float(s["exp"]))
        g["off"].append(first)
        first += synth.ncart(int(s["l"]))
    return {l: {k: np.array(v) for k, v in g.items()} for l, g in sorted(out.items())}
