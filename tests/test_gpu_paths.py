"""GPU parity where the dispatch takes a different kernel or splits the work
differently, at the edges of those rules:

- short lists (one small molecule: block kernels, primitives split over lanes)
  against long lists (copies of it in a batched plan: thread kernels, lists
  ordered by work) and against the oracle, for J+K, the J-engine and the
  gradient;
- primitive screening: tight exponents on two centres, against a plan with
  threshold 0, which drops nothing, and after the atoms move;
- an eager FP64 build captured by the caller before the plan's first build;
- the tensor-core contractions of the exchange-correlation quadrature at the
  edges of their tiles (16 functions, 128 staged, 512 per exact sum), for
  densities whose rows differ by many orders of magnitude, and with
  infinities and NaN, against plain double sums over the oracle's basis values;
- point charges at the edges of the charge chunks.

Tolerances: 1e-10 (J, K, V, density: the parity tolerance of the library), 1e-9
(gradients); two paths of the library against each other 1e-12 of the largest
element (rounding of some 1e4 FP64 additions).
"""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

TOL, GTOL, SAME = 1e-10, 1e-9, 1e-12


@pytest.fixture(scope="module")
def eri():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_14920_gb300.build import build
    build()
    import paper_2406_14920_gb300 as m
    return m


def _t(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, np.float64)).cuda()


def _close(a, b, tol):
    a, b = np.asarray(a), np.asarray(b)
    assert np.abs(a - b).max() <= tol * max(1.0, np.abs(b).max())


@pytest.mark.parametrize("comp", [["2s1p", "1s2p"], ["1s1p1d", "2p1d"], ["1s1p1f"], ["1d1f", "1s"]])
def test_short_and_long_lists(eri, comp):
    b, D = W.small_system(comp, seed=21)
    o = oracle.Oracle(b)
    Q = o.schwarz()
    Jo, Ko = o.jk(D, 1e-12, Q)
    go = o.grad(D, 1e-12, Q)
    one = eri.Plan(b)
    J, K = one.build_jk(_t(D))
    Je, _ = one.build_jk(_t(D), want_k=False)
    g = one.grad(_t(D)).cpu().numpy()
    for x, ref, tol in ((J, Jo, TOL), (K, Ko, TOL), (Je, Jo, TOL)):
        assert np.abs(x.cpu().numpy() - ref).max() < tol
    assert np.abs(g - go).max() < GTOL
    nq = one.stats()["quartets_k"]
    copies = max(2, min(400, 60000 // nq + 1))  # long enough for the thread kernels and the ordered lists
    many = eri.Plan([b] * copies)
    Dp = many.pack([_t(D)] * copies)
    Jm, Km = many.build_jk(Dp)
    Jem, _ = many.build_jk(Dp, want_k=False)
    gm = many.grad(Dp).cpu().numpy().reshape(copies, -1, 3)
    for m in (0, copies // 2, copies - 1):
        _close(many.unpack(Jm)[m].cpu().numpy(), J.cpu().numpy(), SAME)
        _close(many.unpack(Km)[m].cpu().numpy(), K.cpu().numpy(), SAME)
        _close(many.unpack(Jem)[m].cpu().numpy(), Je.cpu().numpy(), SAME)
        _close(gm[m], g, SAME)


def _tight(seed=4):
    """Two atoms 2.5 bohr apart whose contracted s, p and d shells hold exponents up to 1e4."""
    rng = np.random.default_rng(seed)
    shells = []
    for a in range(2):
        for l, e in ((0, [1e4, 300.0, 9.0, 0.4]), (1, [500.0, 20.0, 0.9]), (2, [60.0, 0.8])):
            shells.append((a, l, np.array(e), rng.uniform(0.1, 1.0, len(e))))
    n = np.array([len(s[2]) for s in shells], np.int32)
    off = np.concatenate([[0], np.cumsum(n)[:-1]]).astype(np.int32)
    b = W.Basis(np.array([s[0] for s in shells], np.int32), np.array([s[1] for s in shells], np.int32), n, off,
                np.concatenate([s[2] for s in shells]), np.concatenate([s[3] for s in shells]),
                np.array([[0.0, 0.0, 0.0], [0.3, 0.4, 2.4]]))
    return b, W.density_from_orbitals(rng, b.nbf, 5)


def test_primitive_screening(eri):
    b, D = _tight()
    Dt = _t(D)
    cut, full = eri.Plan(b), eri.Plan(b, thresh=0.0)
    far = b.coords + np.array([[0.0, 0.0, 0.0], [0.0, 0.0, 5.0]])
    for coords in (b.coords, far, b.coords):  # drop primitives, drop more, take them back
        for p in (cut, full):
            p.set_coords(_t(coords))
        o = oracle.Oracle(b.with_coords(coords))
        Q = o.schwarz()
        Jo, Ko = o.jk(D, 0.0, Q)
        for p, thresh in ((cut, 1e-12), (full, 0.0)):
            J, K = p.build_jk(Dt)
            Je, _ = p.build_jk(Dt, want_k=False)
            for x, ref in ((J, Jo), (K, Ko), (Je, Jo)):
                assert np.abs(x.cpu().numpy() - ref).max() < TOL
            assert np.abs(p.grad(Dt).cpu().numpy() - o.grad(D, thresh, Q)).max() < GTOL
    # the screened plan ran fewer primitive quartets over the same lists
    fl = [p.build_jk(Dt) and p.stats()["flops_k"] for p in (cut, full)]
    assert fl[0] < fl[1]


# Lists of 8 items per SM and shorter run a warp per item in the J-engine's large
# classes, longer ones a lane; FP32 items are below the tier bound (1e-5 each, some
# 1e2 per element, 1e-5 of it at most lost with Hermite cancellation): 1e-8.
@pytest.mark.parametrize("mixed,tol", [(False, TOL), (True, 1e-8)])
@pytest.mark.parametrize("copies", [1, 1300])
def test_jengine_large_classes(eri, copies, mixed, tol):
    b, D = W.small_system(["1s1p1d1f", "1f"], seed=31)
    plan = eri.Plan([b] * copies, precision=eri.ERI_MIXED if mixed else eri.ERI_FP64, mixed_tau=1e-5)
    J, _ = plan.build_jk(plan.pack([_t(D)] * copies), want_k=False)
    Jo, _ = oracle.Oracle(b).jk(D)
    for m in (0, copies - 1):
        assert np.abs(plan.unpack(J)[m].cpu().numpy() - Jo).max() < tol


@pytest.mark.parametrize("copies", [1, 120])
def test_captured_before_the_first_build(eri, copies):
    import torch
    b, D = W.small_system(["2s1p1d", "1s1p"], seed=8)
    plan = eri.Plan([b] * copies)
    Dp = plan.pack([_t(D)] * copies)
    J, K = torch.zeros_like(Dp), torch.zeros_like(Dp)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        g.capture_begin()
        plan.build_jk(Dp, J, K)
        g.capture_end()
    torch.cuda.current_stream().wait_stream(s)
    g.replay()
    torch.cuda.synchronize()
    Jo, Ko = oracle.Oracle(b).jk(D)
    for m in (0, copies - 1):
        assert np.abs(plan.unpack(J)[m].cpu().numpy() - Jo).max() < TOL
        assert np.abs(plan.unpack(K)[m].cpu().numpy() - Ko).max() < TOL


def _s_basis(n, seed=2):
    """n diffuse s functions and as many p and d as reach n exactly, on 3 atoms: every block holds all of them."""
    rng = np.random.default_rng(seed)
    ls, left = [], n
    while left:
        l = [2, 1, 0][len(ls) % 3]
        if W.ncart(l) > left:
            l = 0
        ls.append(l)
        left -= W.ncart(l)
    k = len(ls)
    return W.Basis(np.arange(k, dtype=np.int32) % 3, np.array(ls, np.int32), np.ones(k, np.int32),
                   np.arange(k, dtype=np.int32), np.exp(rng.uniform(np.log(0.08), np.log(0.6), k)),
                   np.ones(k), np.array([[0.0, 0.0, 0.0], [1.5, 0.2, 0.0], [-0.3, 1.6, 0.4]]))


def _ao(b, pts):
    """phi [G, n] and grad phi [G, n, 3] of the oracle"""
    o = oracle.Oracle(b)
    r = [o.xc_ao(p) for p in pts]
    return np.array([x[0] for x in r]), np.array([x[1].T for x in r])


@pytest.mark.parametrize("n", [1, 7, 16, 17, 64, 65, 127, 129, 300, 512, 513, 530])
def test_xc_contraction_edges(eri, n):
    b = _s_basis(n)
    assert b.nbf == n
    rng = np.random.default_rng(n)
    D = rng.standard_normal((n, n)) / n
    scale = np.exp(rng.uniform(-12.0, 2.0, n))  # rows over six orders of magnitude
    D = (D + D.T) * np.sqrt(np.outer(scale, scale))
    plan = eri.Plan(b)
    plan.xc_grid(4, 4)
    pts, w = (x.cpu().numpy() for x in plan.xc_get_grid())
    phi, dphi = _ao(b, pts)
    rho, grad = (x.cpu().numpy() for x in plan.xc_density(_t(D)))
    X = phi @ D
    ro, go = (phi * X).sum(1), 2.0 * np.einsum("gm,gmd->gd", X, dphi)
    assert np.abs(rho - ro).max() < TOL * max(1.0, np.abs(ro).max())
    assert np.abs(grad - go).max() < TOL * max(1.0, np.abs(go).max())
    vr, vg = rng.standard_normal(len(w)), rng.standard_normal((len(w), 3))
    Z = w[:, None] * (0.5 * vr[:, None] * phi + np.einsum("gd,gmd->gm", vg, dphi))
    Vo = Z.T @ phi
    Vo = Vo + Vo.T
    V = plan.xc_matrix(_t(vr), _t(vg)).cpu().numpy()
    assert np.abs(V - Vo).max() < TOL * max(1.0, np.abs(Vo).max())
    assert np.array_equal(V, V.T)


def test_xc_infinities_and_nan(eri):
    n = 40
    b = _s_basis(n)
    rng = np.random.default_rng(1)
    D = rng.standard_normal((n, n))
    D = D + D.T
    plan = eri.Plan(b)
    plan.xc_grid(3, 4)
    pts, w = (x.cpu().numpy() for x in plan.xc_get_grid())
    phi, dphi = _ao(b, pts)
    Db = D.copy()
    Db[5, 5] = np.nan
    rho, grad = plan.xc_density(_t(Db))
    assert bool(rho.isnan().all()) and bool(grad.isnan().all())  # every block holds function 5
    Db[5, 5] = np.inf
    rho, _ = plan.xc_density(_t(Db))
    with np.errstate(invalid="ignore"):
        ro = (phi * (phi @ Db)).sum(1)
    assert np.array_equal(np.isnan(rho.cpu().numpy()), np.isnan(ro))
    assert np.array_equal(np.isposinf(rho.cpu().numpy()), np.isposinf(ro))
    vr, vg = rng.standard_normal(len(w)), np.zeros((len(w), 3))
    vr[3] = np.nan
    assert bool(plan.xc_matrix(_t(vr), _t(vg)).isnan().all())
    vr[3] = 0.0  # the plan is as good as before
    Z = w[:, None] * 0.5 * vr[:, None] * phi
    Vo = Z.T @ phi
    V = plan.xc_matrix(_t(vr), _t(vg)).cpu().numpy()
    assert np.abs(V - Vo - Vo.T).max() < TOL * max(1.0, np.abs(Vo).max())
    zero, gzero = plan.xc_density(_t(np.zeros((n, n))))
    assert float(zero.abs().max()) == 0.0 and float(gzero.abs().max()) == 0.0


@pytest.mark.parametrize("nc", [1, 15, 16, 17, 33, 300])
def test_charge_chunks(eri, nc):
    b, D = W.small_system(["1s1p1d1f", "2s1p"], seed=3)
    rng = np.random.default_rng(nc)
    q, C = rng.uniform(-1.0, 1.0, nc), b.coords.mean(0) + rng.normal(0.0, 4.0, (nc, 3))
    C[0] = b.coords[0]  # a charge on a nucleus
    o = oracle.Oracle(b)
    plan = eri.Plan(b)
    V = plan.nuclear(_t(q), _t(C)).cpu().numpy()
    assert np.abs(V - o.nuclear(q, C)).max() < TOL
    gR, gC = plan.nuclear_grad(_t(D), _t(q), _t(C))
    oR, oC = o.nuclear_grad(D, q, C)
    assert np.abs(gR.cpu().numpy() - oR).max() < GTOL and np.abs(gC.cpu().numpy() - oC).max() < GTOL
    g2, none = plan.nuclear_grad(_t(D), _t(q), _t(C), want_charges=False)
    assert none is None and np.abs(g2.cpu().numpy() - oR).max() < GTOL
