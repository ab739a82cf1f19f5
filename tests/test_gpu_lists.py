"""GPU tests of the lists that the builds run over:

- lists frozen at one geometry while the atoms move far apart: shell pairs that
  stay listed although none of their primitive pairs is above the screening
  bound any more, in every kernel (J+K, J-engine, gradient; FP64 and mixed
  precision; short lists and lists ordered by work), against the oracle on the
  same frozen lists;
- deterministic mixed J-only builds: bit for bit the same from call to call and
  in graph replays, over compacted lists of several runs (their order is not
  fixed);
- deterministic FP64 builds over lists that have grown beyond the plan's order
  lists: the same bits before and after those lists are made larger;
- an FP64 build captured by the caller over grown lists, replayed after other
  builds of the plan;
- tier lists taken once: mixed builds over shorter lists, or after a graph build,
  allocate nothing more and can be captured;
- short lists whose items are split over lanes: an item is added a few times at
  most, as the rounding of fixed-point sums shows, and every primitive once.

Tolerances: 1e-10 (J, K) and 1e-9 (gradients), the parity tolerances of the
library.  Mixed precision with a tier bound of 1e-7: an FP32 quartet is at most
1e-7 and off by at most 1e-5 of it (rounding 6e-8 times Hermite cancellation),
some 1e3 of them per element: 1e-9, taken as 1e-8; a derivative brings a factor
2 sqrt(p) of up to 10: 1e-7.
"""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

THRESH = 1e-12


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


def _basis(shells, coords, seed=5):
    """shells: (atom, l, exponents)"""
    rng = np.random.default_rng(seed)
    n = np.array([len(s[2]) for s in shells], np.int32)
    off = np.concatenate([[0], np.cumsum(n)[:-1]]).astype(np.int32)
    return W.Basis(np.array([s[0] for s in shells], np.int32), np.array([s[1] for s in shells], np.int32), n, off,
                   np.concatenate([np.asarray(s[2], float) for s in shells]),
                   rng.uniform(0.3, 1.0, int(n.sum())), np.asarray(coords, float))


# single tight primitives of every angular momentum beside one diffuse s shell per
# atom; contracted s and p shells (lists ordered by work in FP64 builds too)
_SINGLE = [(a, l, [e + 0.5 * a]) for a in range(2) for l, e in ((0, 0.4), (0, 5.0), (1, 5.0), (2, 6.0), (3, 7.0))]
_CONTRACTED = [(a, l, e) for a in range(2) for l, e in ((0, [0.4]), (0, [9.0, 4.0]), (1, [8.0, 4.5]))]


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("shells,copies", [(_SINGLE, 1), (_SINGLE, 3), (_CONTRACTED, 1), (_CONTRACTED, 4000)])
def test_frozen_lists_with_atoms_pulled_apart(eri, shells, copies, mixed):
    near = np.array([[0.0, 0.0, 0.0], [0.2, 0.3, 0.9]])
    far = near + np.array([[0.0, 0.0, 0.0], [1.0, 2.0, 6.0]])
    b = _basis(shells, near)
    D = W.density_from_orbitals(np.random.default_rng(1), b.nbf, 4)
    plan = eri.Plan([b] * copies, thresh=THRESH, precision=eri.ERI_MIXED if mixed else eri.ERI_FP64, mixed_tau=1e-7)
    plan.set_coords(_t(np.concatenate([far] * copies)), freeze_lists=True)
    # the case: every pair is listed, the tight ones on two centres (exponents 4 and more: exp(-2 R^2)) are nothing
    lists = plan.lists()
    assert lists["sig"].all() and np.exp(-2.0 * ((far[1] - far[0]) ** 2).sum()) < 1e-40
    o = oracle.Oracle(b.with_coords(far))
    Q = lists["Q"][:b.nshell * (b.nshell + 1) // 2]
    Jo, Ko = o.jk(D, THRESH, Q)
    go = o.grad(D, THRESH, Q)
    Dp = plan.pack([_t(D)] * copies)
    tol, gtol = (1e-8, 1e-7) if mixed else (1e-10, 1e-9)
    for _ in range(2):
        J, K = plan.build_jk(Dp)
        Je, _ = plan.build_jk(Dp, want_k=False)
        g = plan.grad(Dp, precision=eri.ERI_MIXED if mixed else eri.ERI_FP64).cpu().numpy().reshape(copies, -1, 3)
        for m in {0, copies // 2, copies - 1}:
            for x, ref in ((J, Jo), (K, Ko), (Je, Jo)):
                assert np.abs(plan.unpack(x)[m].cpu().numpy() - ref).max() < tol
            assert np.abs(g[m] - go).max() < gtol


@pytest.mark.parametrize("copies", [3, 60])
def test_deterministic_mixed_j_engine(eri, copies):
    import torch
    b, D = W.small_system(["2s2p1d1f", "1s1p1d"], seed=13)
    plan = eri.Plan([b] * copies, precision=eri.ERI_MIXED, mixed_tau=1e-2, deterministic=True)
    Dp = plan.pack([_t(D)] * copies)
    J = plan.build_jk(Dp, want_k=False)[0].clone()
    assert plan.stats()["quartets_j_fp32"] > 0
    for _ in range(5):
        assert torch.equal(plan.build_jk(Dp, want_k=False)[0], J)
    Jg = torch.empty_like(J)
    for _ in range(2):
        plan.build_jk_graph(Dp, Jg, None)
        assert torch.equal(Jg, J)
    plan.check()


def _s_atoms(counts, nprim, seed=11):
    """counts[a] s shells of nprim primitives on atom a, atoms 1.5 bohr apart in a row."""
    rng = np.random.default_rng(seed)
    atoms = np.repeat(np.arange(len(counts)), counts)
    return _basis([(a, 0, np.exp(rng.uniform(np.log(0.2), np.log(3.0), nprim))) for a in atoms],
                  [[0.0, 0.0, 1.5 * a] for a in range(len(counts))], seed)


def test_deterministic_builds_do_not_depend_on_the_order_lists(eri):
    import torch
    b, copies = _s_atoms([15, 5], 2), 5
    D = W.density_from_orbitals(np.random.default_rng(3), b.nbf, 4)
    apart = b.coords + np.array([[0.0, 0.0, 0.0], [0.0, 0.0, 60.0]])
    plan = eri.Plan([b.with_coords(apart)] * copies, deterministic=True)  # long enough to be ordered by work
    n0 = plan.stats()["quartets_k"]
    plan.set_coords(_t(np.concatenate([b.coords] * copies)))
    assert n0 >= 256 * 152 and plan.stats()["quartets_k"] > 2 * n0  # (256 per SM are ordered)
    Dp = plan.pack([_t(D)] * copies)
    J, K = (x.clone() for x in plan.build_jk(Dp))
    Jg, Kg = torch.empty_like(J), torch.empty_like(K)
    plan.build_jk_graph(Dp, Jg, Kg)  # makes the lists as long as the items
    assert torch.equal(Jg, J) and torch.equal(Kg, K)
    J2, K2 = plan.build_jk(Dp)
    assert torch.equal(J2, J) and torch.equal(K2, K)
    Jo, Ko = oracle.Oracle(b).jk(D)
    assert np.abs(plan.unpack(J)[0].cpu().numpy() - Jo).max() < 1e-10
    assert np.abs(plan.unpack(K)[0].cpu().numpy() - Ko).max() < 1e-10


def _captured(build):
    import torch
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        g.capture_begin()
        try:
            build()
        finally:
            g.capture_end()
    torch.cuda.current_stream().wait_stream(s)
    return g


def test_captured_build_outlives_other_builds(eri):
    import torch
    b, copies = _s_atoms([15, 5], 2), 5
    D = W.density_from_orbitals(np.random.default_rng(3), b.nbf, 4)
    apart = b.coords + np.array([[0.0, 0.0, 0.0], [0.0, 0.0, 60.0]])
    plan = eri.Plan([b.with_coords(apart)] * copies)  # holds order lists
    plan.set_coords(_t(np.concatenate([b.coords] * copies)))  # longer lists
    Dp = plan.pack([_t(D)] * copies)
    J, K = torch.zeros_like(Dp), torch.zeros_like(Dp)
    g = _captured(lambda: plan.build_jk(Dp, J, K))
    Jg, Kg = torch.empty_like(J), torch.empty_like(K)
    for precision in (eri.ERI_FP64, eri.ERI_MIXED):
        plan.build_jk_graph(Dp, Jg, Kg, precision=precision)
        plan.build_jk(Dp, Jg, Kg, precision=precision)
    plan.grad(Dp, precision=eri.ERI_MIXED)
    g.replay()
    torch.cuda.synchronize()
    Jo, Ko = oracle.Oracle(b).jk(D)
    for m in (0, copies - 1):
        assert np.abs(plan.unpack(J)[m].cpu().numpy() - Jo).max() < 1e-10
        assert np.abs(plan.unpack(K)[m].cpu().numpy() - Ko).max() < 1e-10


def test_tier_lists_are_taken_once(eri):
    import torch
    b, copies = _s_atoms([10, 10], 1), 64
    D = W.density_from_orbitals(np.random.default_rng(3), b.nbf, 4)
    plan = eri.Plan([b] * copies, precision=eri.ERI_MIXED)
    Dp = plan.pack([_t(D)] * copies)
    J, K = torch.empty_like(Dp), torch.empty_like(Dp)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    f0 = free()
    plan.build_jk(Dp, J, K)  # long lists: fewer than 16 streams
    f1 = free()
    assert 0 < f0 - f1 < 544 << 20
    plan.build_jk(Dp, J, K, thresh=0.3)  # short lists
    plan.grad(Dp, precision=eri.ERI_MIXED)
    plan.build_jk(Dp, J, None)
    assert abs(free() - f1) < 16 << 20
    apart = np.concatenate([b.coords + np.array([[0.0, 0.0, 0.0], [0.0, 0.0, 60.0]])] * copies)
    plan.set_coords(_t(apart))
    J2, K2 = torch.zeros_like(J), torch.zeros_like(K)
    g = _captured(lambda: plan.build_jk(Dp, J2, K2))
    plan.build_jk(Dp, J, K)
    g.replay()
    torch.cuda.synchronize()
    assert float((J - J2).abs().max()) < 1e-10 and float((K - K2).abs().max()) < 1e-10


def test_mixed_build_captured_after_a_graph_build(eri):
    import torch
    b, D = W.small_system(["2s1p1d", "1s1p"], seed=8)
    plan = eri.Plan(b, precision=eri.ERI_MIXED)
    Dt = _t(D)
    J, K = torch.empty_like(Dt), torch.empty_like(Dt)
    plan.build_jk_graph(Dt, J, K)
    J2, K2 = torch.zeros_like(J), torch.zeros_like(K)
    _captured(lambda: plan.build_jk(Dt, J2, K2)).replay()
    torch.cuda.synchronize()
    assert float((J - J2).abs().max()) < 1e-10 and float((K - K2).abs().max()) < 1e-10


# A deterministic build rounds every addition to 2^-46, so its error shows how often
# an item is added.  A plan that takes a share of the work keeps whole items: two
# shares together are the reference.  A split item is added once per group of lanes
# (three of them cover 81 primitive quartets) or per bra primitive in the block
# kernels, nine times at most: at most three times the rms error, and four with the
# scatter of small matrices (81 additions: nine times).
@pytest.mark.parametrize("comp", [["2s1p", "2s1p"], ["2s1p", "1s"], ["1s1p", "1s1p"], ["1s1p1d", "1s1p"]])
def test_split_items_are_added_a_few_times_at_most(eri, comp):
    b, D = W.small_system(comp, seed=17)
    plan = eri.Plan(b, thresh=0.0, deterministic=True)
    split = [x.cpu().numpy() for x in plan.build_jk(_t(D))]
    whole = 0.0
    for shard in range(2):
        plan.set_shard(shard, 2)
        whole = whole + np.array([x.cpu().numpy() for x in plan.build_jk(_t(D))])
    ref = np.array(oracle.Oracle(b).jk(D, 0.0))
    assert np.abs(split - ref).max() < 1e-10
    rms = [np.sqrt(((x - ref) ** 2).mean()) for x in (split, whole)]
    assert rms[0] < 4.0 * rms[1]
