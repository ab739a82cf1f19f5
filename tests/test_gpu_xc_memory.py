"""Memory of the exchange-correlation grid beside the caller's cap: the digits of
the density (16 nbf^2 bytes), the partial sums of V (at most 1 GiB whatever the
number of functions) and the function lists of the blocks; and V summed over as
few parts as fit, against the oracle.
"""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eri():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_14920_gb300.build import build
    build()
    import paper_2406_14920_gb300 as m
    return m


def test_partial_sums_take_at_most_a_gibibyte(eri):
    import torch
    ns, cap = 800, 64 << 20  # f shells: 8000 functions, 512 MB per half matrix
    rng = np.random.default_rng(6)
    b = W.Basis((np.arange(ns) % 3).astype(np.int32), np.full(ns, 3, np.int32), np.ones(ns, np.int32),
                np.arange(ns, dtype=np.int32), np.exp(rng.uniform(np.log(0.3), np.log(3.0), ns)), np.ones(ns),
                np.array([[0.0, 0.0, 0.0], [1.9, 0.2, 0.0], [-0.3, 2.1, 0.4]]))
    n, natom, nrad, nt = b.nbf, 3, 32, 12
    plan = eri.Plan(b, thresh=1e6)  # no quartets: the plan's own lists are not the point
    torch.cuda.synchronize()
    f0 = torch.cuda.mem_get_info()[0]
    G = plan.xc_grid(nrad, nt, cap_bytes=cap)
    torch.cuda.synchronize()
    used = f0 - torch.cuda.mem_get_info()[0]
    st = plan.xc_stats()
    assert st["nblock"] > 3 * 256  # four parts and more, if memory were no object
    lists = st["nblock"] * (4 * n + 8 * ns + 16) + G * 12 * 8
    assert used < 16 * n * n + (1 << 30) + cap + lists + (64 << 20)
    vr = np.zeros(G)
    sample = rng.integers(0, G, 500)
    vr[sample] = rng.standard_normal(500)
    V = plan.xc_matrix(torch.from_numpy(vr).cuda(), torch.zeros((G, 3), dtype=torch.float64, device="cuda"))
    assert bool((V == V.T).all())
    mn = rng.integers(0, n, (40, 2))
    pts, w = (x.cpu().numpy() for x in plan.xc_get_grid())
    u = np.unique(sample)
    o = oracle.Oracle(b)
    phi = np.array([o.xc_ao(p)[0] for p in pts[u]])
    z = (w[u] * vr[u])[:, None] * phi
    ref = np.einsum("gk,gk->k", z[:, mn[:, 0]], phi[:, mn[:, 1]])
    got = V[torch.from_numpy(mn[:, 0]).cuda(), torch.from_numpy(mn[:, 1]).cuda()].cpu().numpy()
    assert np.abs(got - ref).max() < 1e-10 * max(1.0, np.abs(ref).max())
