"""The work a user of this library has it do, as measurable cases.

Every case goes through the Python binding (``Plan``, ``jk_energy``).  The
molecules are the synthetic ones of this repository: light atoms 2s1p (5 basis
functions), heavy atoms 3s2p1d1f (25) or 4s3p2d1f (35), placed at random at a
density of one atom per 70 cubic bohr with distances of at least 2 bohr, and
random orthonormal orbitals for the density.  A case names the composition;
the seed draws geometry, exponents, coefficients, orbitals and charges.

``exact`` recomputes the outputs in 64 bits with plain torch (unscreened
McMurchie-Davidson integrals with a Boys series, automatic differentiation for
the gradients, dense quadrature sums); it shares nothing with the library.
"""
import math

import numpy as np
import torch

import paper_2406_14920_gb300 as eri

FP64, MIXED = eri.ERI_FP64, eri.ERI_MIXED


def _case(name, kind, light, heavy, shells="4s3p2d1f", **more):
    c = {"name": name, "kind": kind, "light": light, "heavy": heavy, "shells": shells}
    c.update(more)
    return c


def listed():
    return [
        # a diatomic of light atoms: the latency of one SCF iteration's J and K
        _case("jk_tiny", "jk", 2, 0, precision=FP64),
        # three heavy atoms, 75 functions: every class pair up to (ff|ff) with few quartets each
        _case("jk_small", "jk", 0, 3, "3s2p1d1f", precision=FP64),
        # an ordinary organic molecule in plain FP64
        _case("jk_medium", "jk", 10, 5, precision=FP64),
        # 60 atoms, 900 functions, mixed precision: the workload the benchmark quotes
        _case("jk_large_mixed", "jk", 40, 20, precision=MIXED),
        # a batch of small molecules in one plan, replayed as a CUDA graph (high-throughput runs)
        _case("jk_batch_graph", "batch", 7, 3, precision=MIXED, molecules=7),
        # exchange of erf(omega r)/r alone, as a range-separated functional asks for beside its Coulomb build
        _case("k_longrange_mixed", "jk", 17, 9, precision=MIXED, omega=0.3, want_j=False),
        # Coulomb alone through the J-engine (a functional without exact exchange)
        _case("j_engine", "jk", 9, 4, precision=FP64, want_k=False),
        # one geometry-optimisation step of a water-sized molecule: move atoms, energy, all derivatives
        _case("step_small", "step", 2, 1, precision=FP64),
        # nuclear gradient of a medium molecule in mixed precision
        _case("grad_mixed", "grad", 6, 3, precision=MIXED),
        # QM/MM: the field of a few thousand point charges and its forces on atoms and charges
        _case("qmmm", "charges", 8, 4, charges=3001),
        # exchange-correlation of a small molecule on a grid with ragged blocks
        _case("xc_small", "xc", 5, 2, "3s2p1d1f", nrad=27, ntheta=14, functional=eri.ERI_XC_SLATER),
        # exchange-correlation at the benchmark's size, gradient-corrected
        _case("xc_large", "xc", 40, 20, nrad=32, ntheta=16, functional=eri.ERI_XC_B88),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["jk", "jk", "jk", "jk_mixed", "jk_mixed", "batch", "step", "grad", "charges", "xc", "xc"])
    shells = rng.choice(["3s2p1d1f", "4s3p2d1f"])
    if kind == "jk":  # FP64: up to about 250 functions
        heavy = rng.randint(0, 5)
        c = _case("", "jk", _log(rng, 1, 12), heavy, shells, precision=FP64)
        c.update(rng.choice([{}, {}, {"want_k": False}, {"want_j": False, "omega": 0.3}, {"deterministic": True}]))
    elif kind == "jk_mixed":
        heavy = _log(rng, 2, 18)
        c = _case("", "jk", rng.randint(heavy, 2 * heavy), heavy, shells, precision=MIXED)
        c.update(rng.choice([{}, {}, {"want_k": False}, {"omega": 0.4}, {"density_screen": True}]))
    elif kind == "batch":
        c = _case("", "batch", rng.randint(3, 9), rng.randint(1, 3), shells, precision=MIXED, molecules=rng.randint(2, 9))
    elif kind == "step":
        c = _case("", "step", rng.randint(1, 5), 1, shells, precision=FP64)
    elif kind == "grad":
        c = _case("", "grad", rng.randint(2, 8), rng.randint(1, 3), shells, precision=MIXED)
    elif kind == "charges":
        c = _case("", "charges", rng.randint(2, 10), rng.randint(1, 5), shells, charges=_log(rng, 30, 5000))
    else:
        heavy = _log(rng, 1, 16)
        c = _case("", "xc", rng.randint(heavy, 2 * heavy), heavy, shells, nrad=rng.randint(15, 32),
                  ntheta=2 * rng.randint(4, 8), functional=rng.choice([eri.ERI_XC_SLATER, eri.ERI_XC_B88]))
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _ncart(l):
    return (l + 1) * (l + 2) // 2


class _Basis:
    """What ``Plan`` reads: shells in user order with exponents and raw coefficients."""

    def __init__(self, shells, coords):
        self.shell_atom = np.asarray([s[0] for s in shells], np.int32)
        self.shell_l = np.asarray([s[1] for s in shells], np.int32)
        self.shell_nprim = np.asarray([len(s[2]) for s in shells], np.int32)
        self.shell_prim_offset = np.concatenate([[0], np.cumsum(self.shell_nprim)[:-1]]).astype(np.int32)
        self.exps = np.concatenate([s[2] for s in shells])
        self.coefs = np.concatenate([s[3] for s in shells])
        self.coords = coords
        self.nshell, self.natom = len(shells), len(coords)
        self.nbf = int(sum(_ncart(int(l)) for l in self.shell_l))


def _parse(shells):
    return [int(n) for n in shells[0::2]], ["spdf".index(l) for l in shells[1::2]]


def _molecule(rng, light, heavy, shells):
    n = light + heavy
    side, pts = max(4.0, (n * 70.0) ** (1 / 3)), []
    while len(pts) < n:
        x = rng.uniform(0.0, side, size=3)
        if all(np.linalg.norm(x - p) >= 2.0 for p in pts):
            pts.append(x)
    is_heavy = np.zeros(n, bool)
    is_heavy[rng.permutation(n)[:heavy]] = True
    out = []
    for a in range(n):
        for count, l in zip(*_parse(shells if is_heavy[a] else "2s1p")):
            for _ in range(count):
                k, lo, hi = (3, 0.1, 50.0) if l < 2 else (1, 0.3, 3.0)
                out.append((a, l, np.exp(rng.uniform(math.log(lo), math.log(hi), k)), rng.uniform(0.1, 1.0, k)))
    return _Basis(out, np.asarray(pts))


def _density(rng, nbf):
    q, _ = np.linalg.qr(rng.standard_normal((nbf, max(1, round(nbf / 7.5)))))
    d = q @ q.T
    return np.ascontiguousarray(0.5 * (d + d.T))


def _inputs(case, seed):
    rng = np.random.default_rng([int(seed) & 0xFFFFFFFF, 14920])
    mols = [_molecule(rng, case["light"] + m % 4, case["heavy"] + m % 2, case["shells"])  # a batch is uneven
            for m in range(case.get("molecules", 1))]
    dens = [_density(rng, m.nbf) for m in mols]
    q = xyz = None
    if case["kind"] == "charges":  # a solvent shell around the molecule, neutral on average
        nc, c = case["charges"], mols[0].coords.mean(0)
        r = rng.uniform(6.0, 40.0, nc) + np.abs(mols[0].coords - c).max()
        v = rng.standard_normal((nc, 3))
        xyz = c + r[:, None] * v / np.linalg.norm(v, axis=1, keepdims=True)
        xyz[:mols[0].natom] = mols[0].coords[:nc]  # the nuclei are charges too
        q = rng.uniform(-0.8, 0.8, nc)
        q[:mols[0].natom] = -rng.integers(1, 9, min(nc, mols[0].natom))
    return mols, dens, q, xyz


class _State:
    pass


def prepare(case, seed):
    mols, dens, q, xyz = _inputs(case, seed)
    st = _State()
    st.case = case
    kind = case["kind"]
    opts = {"precision": case.get("precision", FP64)}  # mixed: the default tier bound
    for k in ("deterministic", "density_screen"):
        if case.get(k):
            opts[k] = True
    st.plan = eri.Plan(mols if kind == "batch" else mols[0], **opts)
    if case.get("omega"):
        st.plan.set_omega(case["omega"])
    if kind == "batch":
        st.D = st.plan.pack([torch.from_numpy(d).cuda() for d in dens])
        st.J, st.K = torch.empty_like(st.D), torch.empty_like(st.D)
    else:
        st.D = torch.from_numpy(dens[0]).cuda()
    if kind == "step":
        st.R = torch.from_numpy(mols[0].coords).cuda().requires_grad_()
        st.D.requires_grad_()
    if kind == "charges":
        st.q, st.xyz = torch.from_numpy(q).cuda(), torch.from_numpy(xyz).cuda()
    if kind == "xc":
        st.plan.xc_grid(case["nrad"], case["ntheta"])
    return st


def run(st):
    case, plan = st.case, st.plan
    kind = case["kind"]
    if kind == "jk":
        J, K = plan.build_jk(st.D, want_j=case.get("want_j", True), want_k=case.get("want_k", True))
        return {k: v for k, v in (("J", J), ("K", K)) if v is not None}
    if kind == "batch":
        J, K = plan.build_jk_graph(st.D, st.J, st.K)
        return {"J": J, "K": K}
    if kind == "step":
        E = eri.jk_energy(st.R, st.D, plan)
        gR, gD = torch.autograd.grad(E, (st.R, st.D))
        return {"E": E, "gR": gR, "gD": gD}
    if kind == "grad":
        return {"gR": plan.grad(st.D, precision=case["precision"])}
    if kind == "charges":
        V = plan.nuclear(st.q, st.xyz)
        gR, gC = plan.nuclear_grad(st.D, st.q, st.xyz)
        return {"V": V, "gR": gR, "gC": gC}
    E, V = plan.xc(st.D, functional=case["functional"])
    return {"E": E, "V": V}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

def _nherm(n):
    return (n + 1) * (n + 2) * (n + 3) // 6 if n >= 0 else 0


def _carts(l):
    return [(l - r, r - z, z) for r in range(l + 1) for z in range(r + 1)]


def _terms(la, lb):
    return sum((i[0] + j[0] + 1) * (i[1] + j[1] + 1) * (i[2] + j[2] + 1) for i in _carts(la) for j in _carts(lb))


def _r_flops(L):
    return 2.0 * (L + 1) + 20.0 + sum(3.0 * (_nherm(L - m) - 1) for m in range(L))


def _pair_list(b):
    """(l1, l2, primitives, estimated Schwarz bound) of every shell pair, higher l first;
    the bound is that of s functions with the same exponents."""
    out = []
    for x in range(b.nshell):
        for y in range(x + 1):
            i, j = (x, y) if b.shell_l[x] >= b.shell_l[y] else (y, x)
            oi, oj, ni, nj = b.shell_prim_offset[i], b.shell_prim_offset[j], b.shell_nprim[i], b.shell_nprim[j]
            a, c = b.exps[oi:oi + ni, None], b.exps[None, oj:oj + nj]
            p = a + c
            r2 = float(((b.coords[b.shell_atom[i]] - b.coords[b.shell_atom[j]]) ** 2).sum())
            k = ((2 * a / math.pi) ** 0.75 * (2 * c / math.pi) ** 0.75 * np.exp(-a * c / p * r2) * math.pi ** 1.25 *
                 2 ** 0.25 / p ** 1.25)
            out.append((int(b.shell_l[i]), int(b.shell_l[j]), int(ni * nj), float(k.sum())))
    return out


def work(case):
    mols, dens, q, _ = _inputs(case, 1)
    nn = sum(m.nbf ** 2 for m in mols)
    kind = case["kind"]
    if kind == "xc":
        pts = mols[0].natom * case["nrad"] * 2 * case["ntheta"] ** 2
        near = min(1.0, 45.0 / mols[0].natom)  # share of the functions that reach a point
        nb = mols[0].nbf * near
        return {"bytes": 8.0 * (2 * nn + 4 * pts), "flops": pts * (4.0 * nb * nb + 60.0 * nb)}
    if kind == "charges":
        nc, fl = case["charges"], 0.0
        for l1, l2, k, _ in _pair_list(mols[0]):
            L = l1 + l2
            per = _r_flops(L) + 2 * _nherm(L)                       # the matrix
            per += _r_flops(L + 1) + 6 * (_nherm(L) + _nherm(L + 1))  # both gradients from one R
            fl += k * nc * per
        return {"bytes": 8.0 * (2 * nn + 7 * nc), "flops": fl}
    flops = 0.0
    deriv = kind in ("step", "grad")
    want_j, want_k = case.get("want_j", True), case.get("want_k", True)
    for m in mols:
        cls = {}
        for l1, l2, k, s in _pair_list(m):
            cls.setdefault((l1, l2), []).append((s, k))
        qmax = max(s for v in cls.values() for s, _ in v)
        keys = sorted(cls)
        for v in cls.values():
            v.sort()
        for X in keys:
            for Y in keys:
                if not deriv and Y > X:
                    continue
                sy = np.asarray([s for s, _ in cls[Y]])
                ky = np.concatenate([np.cumsum([k for _, k in cls[Y]][::-1])[::-1], [0]])
                sx, kx = np.asarray([s for s, _ in cls[X]]), np.asarray([k for _, k in cls[X]])
                keep = sx * qmax >= 1e-12
                sx, kx = sx[keep], kx[keep]
                at = np.searchsorted(sy, 1e-12 / np.maximum(sx, 1e-300))
                half = 0.5 if (X == Y and not deriv) else 1.0
                nq, npq = half * float((len(sy) - at).sum()), half * float((kx * ky[at]).sum())
                nbp = half * float((kx * (len(sy) - at)).sum())
                (la, lb), (lc, ld) = X, Y
                L = la + lb + lc + ld + (1 if deriv else 0)
                nab, ncd = _ncart(la) * _ncart(lb), _ncart(lc) * _ncart(ld)
                if want_j and not want_k and not deriv:  # Hermite Coulomb
                    flops += npq * (_r_flops(L) + 4.0 * _nherm(la + lb) * _nherm(lc + ld))
                    continue
                flops += npq * (_r_flops(L) + 2.0 * _nherm(la + lb + (1 if deriv else 0)) * _terms(lc, ld))
                flops += nbp * 2.0 * ncd * _terms(la, lb) * (3 if deriv else 1)
                flops += nq * nab * ncd * ((8.0 if want_k else 0.0) + (4.0 if want_j else 0.0))
    return {"bytes": 8.0 * nn * (3 if kind != "jk" else 1 + int(want_j) + int(want_k)), "flops": flops}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits, without the library
# ---------------------------------------------------------------------------

_F64 = torch.float64


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _fact2(n):
    return 1.0 if n <= 1 else n * _fact2(n - 2)


class _BoysF(torch.autograd.Function):
    """F_0..F_L at T: the convergent series below 36, erf and upward recursion above."""

    @staticmethod
    def _eval(T, L):
        lo = T.clamp(max=36.0)
        term = torch.full_like(lo, 1.0 / (2 * L + 1))
        top = term.clone()
        for k in range(1, 150):
            term = term * lo * (2.0 / (2 * L + 2 * k + 1))
            top += term
        e = torch.exp(-lo)
        F = [None] * (L + 1)
        F[L] = top * e
        for m in range(L - 1, -1, -1):
            F[m] = (2.0 * lo * F[m + 1] + e) / (2 * m + 1)
        hi = T.clamp(min=36.0)
        eh = torch.exp(-hi)
        g = 0.5 * torch.sqrt(math.pi / hi)
        big = T > 36.0
        for m in range(L + 1):
            F[m] = torch.where(big, g, F[m])
            g = ((2 * m + 1) * g - eh) / (2.0 * hi)
        return F

    @staticmethod
    def forward(ctx, T, L):
        F = _BoysF._eval(T, L + 1)
        ctx.save_for_backward(*F[1:])
        return tuple(F[:L + 1])

    @staticmethod
    def backward(ctx, *g):
        out = None
        for gm, f in zip(g, ctx.saved_tensors):
            if gm is not None:
                out = -gm * f if out is None else out - gm * f
        return out, None


def _herms(n):
    return [(t, u, v) for t in range(n + 1) for u in range(n + 1 - t) for v in range(n + 1 - t - u)]


def _r_table(rho, X, Y, Z, L, scale):
    """{(t,u,v): scale * R^0_tuv} for t+u+v <= L."""
    F = _BoysF.apply(rho * (X * X + Y * Y + Z * Z), L)
    lev = {}
    for m in range(L, -1, -1):
        new = {(0, 0, 0): scale * (-2.0 * rho) ** m * F[m]}
        for t, u, v in _herms(L - m):
            if t + u + v == 0:
                continue
            d = 0 if t else (1 if u else 2)
            lower = [t, u, v]
            lower[d] -= 1
            val = (X, Y, Z)[d] * lev[tuple(lower)]
            if lower[d]:
                k = lower[d]
                lower[d] -= 1
                val = val + k * lev[tuple(lower)]
            new[(t, u, v)] = val
        lev = new
    return lev


def _e1d(PA, PB, o2p, la, lb):
    E = {(0, 0): [torch.ones_like(PA)]}

    def raise_(src, x):
        out = []
        for t in range(len(src) + 1):
            v = x * src[t] if t < len(src) else 0
            if t > 0:
                v = v + o2p * src[t - 1]
            if t + 1 < len(src):
                v = v + (t + 1) * src[t + 1]
            out.append(v)
        return out

    for i in range(la):
        E[(i + 1, 0)] = raise_(E[(i, 0)], PA)
    for i in range(la + 1):
        for j in range(lb):
            E[(i, j + 1)] = raise_(E[(i, j)], PB)
    return E


def _shell_norms(b):
    """c_k (2a/pi)^(3/4) (4a)^(l/2) per primitive, scaled so that the contracted (l,0,0) has unit norm
    (the components' 1/sqrt((2i-1)!!(2j-1)!!(2k-1)!!) comes on top)."""
    out = []
    for s in range(b.nshell):
        o, k, l = b.shell_prim_offset[s], b.shell_nprim[s], int(b.shell_l[s])
        a, c = b.exps[o:o + k], b.coefs[o:o + k]
        ov = (2 * np.sqrt(a[:, None] * a[None]) / (a[:, None] + a[None])) ** (l + 1.5)
        out.append(c / math.sqrt(c @ ov @ c) * (2 * a / math.pi) ** 0.75 * (4 * a) ** (l / 2))
    return out


class _Mol:
    """Normalised shells and the primitive pairs of every pair class, as tensors on `R` (atoms x 3)."""

    def __init__(self, b, R):
        dev = R.device
        norm = _shell_norms(b)
        self.ao = np.concatenate([[0], np.cumsum([_ncart(int(l)) for l in b.shell_l])]).astype(np.int64)
        groups = {}
        for x in range(b.nshell):
            for y in range(x + 1):
                i, j = (x, y) if b.shell_l[x] >= b.shell_l[y] else (y, x)
                key = (int(b.shell_l[i]), int(b.shell_l[j]), int(b.shell_nprim[i] * b.shell_nprim[j]))
                groups.setdefault(key, []).append((i, j))
        T = lambda v, dt=_F64: torch.as_tensor(np.asarray(v), dtype=dt, device=dev)
        self.cls = []
        for (la, lb, npr), prs in sorted(groups.items()):
            ea, eb, cc = [], [], []
            for i, j in prs:
                oi, oj, ni, nj = (int(v) for v in (b.shell_prim_offset[i], b.shell_prim_offset[j],
                                                   b.shell_nprim[i], b.shell_nprim[j]))
                ea.append(np.repeat(b.exps[oi:oi + ni], nj))
                eb.append(np.tile(b.exps[oj:oj + nj], ni))
                cc.append(np.outer(norm[i], norm[j]).reshape(-1))
            ea, eb, cc = T(ea), T(eb), T(cc)  # [pairs, primitives]
            A = R[T([b.shell_atom[i] for i, _ in prs], torch.long)][:, None, :]
            B = R[T([b.shell_atom[j] for _, j in prs], torch.long)][:, None, :]
            p = ea + eb
            P = (ea[..., None] * A + eb[..., None] * B) / p[..., None]
            pref = cc * torch.exp(-ea * eb / p * ((A - B) ** 2).sum(-1))
            E1 = [_e1d(P[..., d] - A[..., d], P[..., d] - B[..., d], 0.5 / p, la, lb) for d in range(3)]
            H = _herms(la + lb)
            comps = [(i, j) for i in _carts(la) for j in _carts(lb)]
            zero = torch.zeros_like(pref)
            rows = []
            for t in H:
                row = []
                for i, j in comps:
                    if any(t[d] > i[d] + j[d] for d in range(3)):
                        row.append(zero)
                        continue
                    f = 1.0
                    for c, l in ((i, la), (j, lb)):
                        f *= math.sqrt(1.0 / (_fact2(2 * c[0] - 1) * _fact2(2 * c[1] - 1) * _fact2(2 * c[2] - 1)))
                    row.append(f * pref * E1[0][(i[0], j[0])][t[0]] * E1[1][(i[1], j[1])][t[1]] *
                               E1[2][(i[2], j[2])][t[2]])
                rows.append(torch.stack(row, -1))
            self.cls.append({"la": la, "lb": lb, "p": p, "P": P, "E": torch.stack(rows, -2), "H": H, "na": _ncart(la), "nb": _ncart(lb),
                             "oa": T([self.ao[i] for i, _ in prs], torch.long),
                             "ob": T([self.ao[j] for _, j in prs], torch.long),
                             "w": T([0.5 if i == j else 1.0 for i, j in prs])})


def _quartets(bra, sl, ket, omega):
    """(ab|cd) of bra pairs `sl` with every ket pair: [bra, ket, ab, cd]."""
    L = bra["la"] + bra["lb"] + ket["la"] + ket["lb"]
    p, P, Eb = bra["p"][sl], bra["P"][sl], bra["E"][sl]
    nb, kb = p.shape
    nk, kk = ket["p"].shape
    pb, pk = p.reshape(-1, 1), ket["p"].reshape(1, -1)
    d = P.reshape(-1, 1, 3) - ket["P"].reshape(1, -1, 3)
    rho = pb * pk / (pb + pk)
    scale = 2 * math.pi ** 2.5 / (pb * pk * torch.sqrt(pb + pk))
    if omega:
        s = omega * omega / (omega * omega + rho)
        rho, scale = rho * s, scale * torch.sqrt(s)
    R = _r_table(rho, d[..., 0], d[..., 1], d[..., 2], L, scale)
    Ek = ket["E"].reshape(nk * kk, len(ket["H"]), -1)
    sign = torch.tensor([(-1.0) ** sum(q) for q in ket["H"]], dtype=_F64, device=p.device)
    Ek = Ek * sign[None, :, None]
    W = []
    for t in bra["H"]:
        M = torch.stack([R[(t[0] + q[0], t[1] + q[1], t[2] + q[2])] for q in ket["H"]], -1)  # [nb kb, nk kk, HQ]
        X = torch.bmm(M.transpose(0, 1), Ek)  # [nk kk, nb kb, cd]
        W.append(X.reshape(nk, kk, nb * kb, -1).sum(1))
    W = torch.stack(W, 1).reshape(nk, len(bra["H"]), nb, kb, -1).permute(2, 3, 1, 0, 4)  # [nb, kb, HP, nk, cd]
    W = W.reshape(nb, kb * len(bra["H"]), -1)
    V = torch.bmm(Eb.reshape(nb, kb * len(bra["H"]), -1).transpose(1, 2), W)  # [nb, ab, nk cd]
    return V.reshape(nb, Eb.shape[-1], nk, -1).permute(0, 2, 1, 3)


def _blocks(mol, doubles, kept=False):
    """(bra class, slice, ket class, same class) in pieces of about `doubles` values of storage;
    kept: what automatic differentiation keeps is counted too."""
    for x, bra in enumerate(mol.cls):
        for y in range(x + 1):
            ket = mol.cls[y]
            L = bra["la"] + bra["lb"] + ket["la"] + ket["lb"]
            per = ket["p"].numel() * bra["p"].shape[1] * (_nherm(L) * (L + 2) / 2 + _nherm(ket["la"] + ket["lb"]) + 30)
            if kept:
                per += ket["p"].numel() * bra["p"].shape[1] * 2 * len(bra["H"]) * len(ket["H"])
            per += len(ket["w"]) * bra["E"].shape[-1] * ket["E"].shape[-1] * 4
            step = max(1, int(doubles / per))
            for i in range(0, len(bra["w"]), step):
                yield bra, slice(i, min(i + step, len(bra["w"]))), ket, x == y


def _take(M, ra, na, rb, nb):
    """blocks M[ra_i + :na, rb_j + :nb] for broadcast index tensors"""
    dev = M.device
    return M[ra[..., None, None] + torch.arange(na, device=dev)[:, None], rb[..., None, None] + torch.arange(nb, device=dev)]


def _add(M, ra, na, rb, nb, v):
    dev = M.device
    r = (ra[..., None, None] + torch.arange(na, device=dev)[:, None]).expand(v.shape)
    c = (rb[..., None, None] + torch.arange(nb, device=dev)).expand(v.shape)
    M.index_put_((r.reshape(-1), c.reshape(-1)), v.reshape(-1), accumulate=True)


def _exact_jk(b, D, omega, want_j, want_k):
    dev = _dev()
    D = torch.from_numpy(D).to(dev)
    mol = _Mol(b, torch.from_numpy(b.coords).to(dev))
    J, K = torch.zeros_like(D), torch.zeros_like(D)
    for bra, sl, ket, same in _blocks(mol, 2e9):
        V = _quartets(bra, sl, ket, omega)
        nb, nk = V.shape[:2]
        na, n2, n3, n4 = bra["na"], bra["nb"], ket["na"], ket["nb"]
        oa, ob, wb = bra["oa"][sl][:, None], bra["ob"][sl][:, None], bra["w"][sl][:, None]
        oc, od, wk = ket["oa"][None], ket["ob"][None], ket["w"][None]
        V = V.reshape(nb, nk, na, n2, n3, n4) * (wb * wk)[..., None, None, None, None]
        oa, ob, oc, od = (v.expand(nb, nk) for v in (oa, ob, oc, od))
        if want_j:
            jab = 2 * torch.einsum("xyabcd,xycd->xab", V, _take(D, oc, n3, od, n4))
            _add(J, oa[:, 0], na, ob[:, 0], n2, jab)
            if not same:
                jcd = 2 * torch.einsum("xyabcd,xyab->ycd", V, _take(D, oa, na, ob, n2))
                _add(J, oc[0], n3, od[0], n4, jcd)
        if want_k:
            Kp = torch.zeros_like(K)
            _add(Kp, oa, na, oc, n3, torch.einsum("xyabcd,xybd->xyac", V, _take(D, ob, n2, od, n4)))
            _add(Kp, oa, na, od, n4, torch.einsum("xyabcd,xybc->xyad", V, _take(D, ob, n2, oc, n3)))
            _add(Kp, ob, n2, oc, n3, torch.einsum("xyabcd,xyad->xybc", V, _take(D, oa, na, od, n4)))
            _add(Kp, ob, n2, od, n4, torch.einsum("xyabcd,xyac->xybd", V, _take(D, oa, na, oc, n3)))
            K += Kp if same else Kp + Kp.T
        del V
    return J + J.T, K


def _exact_grad(b, D):
    """dE/dR of E = 1/2 tr(DJ) - 1/4 tr(DK) by automatic differentiation of the pieces."""
    dev = _dev()
    D = torch.from_numpy(D).to(dev)
    R = torch.from_numpy(b.coords).to(dev).requires_grad_()
    g = torch.zeros_like(R)
    with torch.no_grad():
        pieces = list(_index_blocks(_Mol(b, R.detach()), 3e9))
    mol = _Mol(b, R)
    for c in mol.cls:  # differentiate the pieces to the pair data, then the pair data to the atoms at once
        c["src"] = (c["P"], c["E"])
        c["P"], c["E"] = c["P"].detach().requires_grad_(), c["E"].detach().requires_grad_()
    for x, sl, y, same in pieces:
        bra, ket = mol.cls[x], mol.cls[y]
        V = _quartets(bra, sl, ket, 0.0)
        nb, nk = V.shape[:2]
        na, n2, n3, n4 = bra["na"], bra["nb"], ket["na"], ket["nb"]
        oa, ob = bra["oa"][sl][:, None].expand(nb, nk), bra["ob"][sl][:, None].expand(nb, nk)
        oc, od = ket["oa"][None].expand(nb, nk), ket["ob"][None].expand(nb, nk)
        w = (bra["w"][sl][:, None] * ket["w"][None]) * (1.0 if same else 2.0)
        G = 2.0 * torch.einsum("xyab,xycd->xyabcd", _take(D, oa, na, ob, n2), _take(D, oc, n3, od, n4))
        G -= 0.5 * torch.einsum("xyac,xybd->xyabcd", _take(D, oa, na, oc, n3), _take(D, ob, n2, od, n4))
        G -= 0.5 * torch.einsum("xyad,xybc->xyabcd", _take(D, oa, na, od, n4), _take(D, ob, n2, oc, n3))
        G = G * w[..., None, None, None, None]
        (V.reshape(G.shape) * G).sum().backward()
        del V, G
    for c in mol.cls:
        for src, leaf in zip(c["src"], (c["P"], c["E"])):
            if leaf.grad is not None and src.requires_grad:
                g += torch.autograd.grad(src, R, leaf.grad, retain_graph=True)[0]
    return g


def _index_blocks(mol, doubles):
    at = {id(c): i for i, c in enumerate(mol.cls)}
    for bra, sl, ket, same in _blocks(mol, doubles, kept=True):
        yield at[id(bra)], sl, at[id(ket)], same


def _exact_charges(b, D, q, xyz):
    dev = _dev()
    D, q = torch.from_numpy(D).to(dev), torch.from_numpy(q).to(dev)
    R = torch.from_numpy(b.coords).to(dev).requires_grad_()
    C = torch.from_numpy(xyz).to(dev).requires_grad_()
    V, gR, gC = torch.zeros_like(D), torch.zeros_like(R), torch.zeros_like(C)
    mol = _Mol(b, R)
    for c in mol.cls:
        n, k = c["p"].shape
        L, na, nb = c["la"] + c["lb"], c["na"], c["nb"]
        P, E = c["P"].detach().requires_grad_(), c["E"].detach().requires_grad_()
        step = max(1, int(1.5e9 / (k * len(q) * (_nherm(L) * (L + 2) / 2 + 30))))
        for i in range(0, n, step):
            sl = slice(i, min(n, i + step))
            d = P[sl].reshape(-1, 1, 3) - C[None]
            p = c["p"][sl].reshape(-1, 1)
            T = _r_table(p, d[..., 0], d[..., 1], d[..., 2], L, 2 * math.pi / p * q[None])
            h = torch.stack([T[t].sum(-1) for t in c["H"]], -1)
            blk = torch.einsum("xkh,xkhm->xm", h.reshape(-1, k, len(c["H"])), E[sl]).reshape(-1, na, nb)
            oa, ob, w = c["oa"][sl], c["ob"][sl], c["w"][sl][:, None, None]
            with torch.no_grad():
                _add(V, oa, na, ob, nb, blk * w)
            (2.0 * blk * w * _take(D, oa, na, ob, nb)).sum().backward()
            del T, h, blk, d
        for src, leaf in ((c["P"], P), (c["E"], E)):
            if src.requires_grad:
                gR += torch.autograd.grad(src, R, leaf.grad, retain_graph=True)[0]
    gC = C.grad
    return V + V.T, gR, gC


def _exact_xc(b, D, nrad, ntheta, functional):
    dev = _dev()
    D = torch.from_numpy(D).to(dev)
    R = torch.from_numpy(b.coords).to(dev)
    T = lambda v: torch.as_tensor(np.asarray(v), dtype=_F64, device=dev)
    th = np.arange(1, nrad + 1) * math.pi / (nrad + 1)
    x = np.cos(th)
    r = (1 + x) / (1 - x)
    wr = math.pi / (nrad + 1) * np.sin(th) * r * r * 2 / (1 - x) ** 2
    ct, wt = np.polynomial.legendre.leggauss(ntheta)
    nphi = 2 * ntheta
    ph = 2 * math.pi * (np.arange(nphi) + 0.5) / nphi
    s = np.sqrt(1 - ct * ct)
    u = np.stack([s[:, None] * np.cos(ph), s[:, None] * np.sin(ph), np.repeat(ct[:, None], nphi, 1)], -1).reshape(-1, 3)
    off, wq = T((r[:, None, None] * u[None]).reshape(-1, 3)), T(np.outer(wr, np.repeat(wt * 2 * math.pi / nphi, nphi)).reshape(-1))
    norm = _shell_norms(b)
    ao = np.concatenate([[0], np.cumsum([_ncart(int(l)) for l in b.shell_l])])
    dab = (R[:, None] - R[None]).norm(dim=-1)
    dab.fill_diagonal_(1.0)
    E, V = torch.zeros((), dtype=_F64, device=dev), torch.zeros_like(D)
    na, step = b.natom, 32768
    for a in range(na):
        for i in range(0, len(off), step):
            pts = R[a] + off[i:i + step]
            d = (pts[:, None] - R[None]).norm(dim=-1)
            cell = torch.ones_like(d)
            for B in range(na):
                mu = (d - d[:, B:B + 1]) / dab[:, B]
                for _ in range(3):
                    mu = 1.5 * mu - 0.5 * mu ** 3
                f = 0.5 * (1 - mu)
                f[:, B] = 1.0
                cell *= f
            w = wq[i:i + step] * cell[:, a] / cell.sum(1)
            phi = torch.zeros((4, len(pts), b.nbf), dtype=_F64, device=dev)
            for sh in range(b.nshell):
                v = pts - R[int(b.shell_atom[sh])]
                o, k, l = b.shell_prim_offset[sh], b.shell_nprim[sh], int(b.shell_l[sh])
                al = T(b.exps[o:o + k])
                e = T(norm[sh]) * torch.exp(-al * (v * v).sum(1, keepdim=True))
                e0, e1 = e.sum(1), (e * al).sum(1)
                pw = [torch.ones_like(v)]
                for _ in range(l + 1):
                    pw.append(pw[-1] * v)
                for c, ijk in enumerate(_carts(l)):
                    f = 1.0 / math.sqrt(math.prod(_fact2(2 * n - 1) for n in ijk))
                    g = [pw[ijk[t]][:, t] for t in range(3)]
                    col = int(ao[sh]) + c
                    phi[0, :, col] = f * g[0] * g[1] * g[2] * e0
                    for t in range(3):
                        n = ijk[t]
                        dt = -2.0 * pw[n + 1][:, t] * e1
                        if n:
                            dt = dt + n * pw[n - 1][:, t] * e0
                        phi[1 + t, :, col] = f * dt * g[(t + 1) % 3] * g[(t + 2) % 3]
            X = phi[0] @ D
            rho = (phi[0] * X).sum(1).detach()
            grad = 2.0 * (phi[1:] * X).sum(2)
            ok = rho >= 1e-14
            rr = torch.where(ok, rho, torch.ones_like(rho)).requires_grad_()
            gg = torch.where(ok, grad, torch.zeros_like(grad)).requires_grad_()
            if functional == eri.ERI_XC_SLATER:
                eps = -0.75 * (3 / math.pi) ** (1 / 3) * rr ** (4 / 3) + 0.0 * gg.sum()
            else:
                n43 = (0.5 * rr) ** (4 / 3)
                g2 = (gg * gg).sum(0)
                xs = 0.5 * torch.sqrt(torch.where(g2 > 0, g2, torch.ones_like(g2))) / n43
                xs = torch.where(g2 > 0, xs, torch.zeros_like(xs))
                beta = 0.0042
                eps = -2 * n43 * (1.5 * (3 / (4 * math.pi)) ** (1 / 3) + beta * xs * xs / (1 + 6 * beta * xs * torch.asinh(xs)))
            vr, vg = torch.autograd.grad(eps.sum(), (rr, gg))
            m = torch.where(ok, w, torch.zeros_like(w))
            E += (m * eps.detach()).sum()
            Z = (0.5 * m * vr)[:, None] * phi[0]
            for t in range(3):
                Z += (m * vg[t])[:, None] * phi[1 + t]
            V += Z.T @ phi[0]
            del phi, X, Z
    return E.reshape(1), V + V.T


def exact(case, seed):
    mols, dens, q, xyz = _inputs(case, seed)
    b, D, kind = mols[0], dens[0], case["kind"]
    if kind == "jk":
        if b.nbf > 260:
            return None  # minutes without screening
        J, K = _exact_jk(b, D, case.get("omega", 0.0), case.get("want_j", True), case.get("want_k", True))
        return {k: v for k, v, w in (("J", J, case.get("want_j", True)), ("K", K, case.get("want_k", True))) if w}
    if kind == "batch":
        jk = [_exact_jk(m, d, 0.0, True, True) for m, d in zip(mols, dens)]
        return {n: torch.cat([x[i].reshape(-1) for x in jk]) for i, n in ((0, "J"), (1, "K"))}
    if kind == "step":
        J, K = _exact_jk(b, D, 0.0, True, True)
        Dt = torch.from_numpy(D).to(J.device)
        return {"E": 0.5 * (Dt * J).sum() - 0.25 * (Dt * K).sum(), "gR": _exact_grad(b, D), "gD": J - 0.5 * K}
    if kind == "grad":
        return {"gR": _exact_grad(b, D)}
    if kind == "charges":
        V, gR, gC = _exact_charges(b, D, q, xyz)
        return {"V": V, "gR": gR, "gC": gC}
    E, V = _exact_xc(b, D, case["nrad"], case["ntheta"], case["functional"])
    return {"E": E, "V": V}
