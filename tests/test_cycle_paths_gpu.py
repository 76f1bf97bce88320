"""V-cycles where the coarse levels' kernel and the separate launches meet: other
sweep counts than V(3,3), coarse meshes from a few to a thousand macros against
the oracle's cycle, and the same bits from both (needs a GPU)."""
import numpy as np
import pytest

import oracle.multigrid as omg
from inputs import unit_square_mesh, unit_cube_kuhn_mesh

pytestmark = pytest.mark.gpu


def _rhs(h, L):
    rm = h.meshes[L]
    f = np.prod(np.sin(np.pi * rm.coords), axis=1) + 0.1 * np.random.default_rng(L).standard_normal(rm.n_global)
    return omg.poisson_rhs(rm, f)


def _two_cycles(coarse, L, nu1, nu2, kind):
    """Two cycles from zero on the GPU and by the oracle, slot by slot."""
    import torch
    import paper_2305_15116_gb300 as H
    dt = torch.float64 if kind == "f64" else torch.float32
    M = H.Mesh(coarse.coords, coarse.cells).refine(L).solver_setup(L, nu1, nu2)
    h = omg.Hierarchy(coarse.coords, coarse.cells, L)
    b = _rhs(h, L)
    smap = M.dof_map(L)
    u = torch.zeros(len(smap), dtype=dt, device="cuda")
    bd = torch.from_numpy(b[smap]).to("cuda", dt)
    ref = np.zeros_like(b)
    for _ in range(2):
        M.vcycle(L, bd, u)
        ref = h.vcycle(L, ref, b, nu1, nu2)
    got = u.double().cpu().numpy()
    M.close()
    return got, ref[smap]


# per cycle: the tolerances of the V(3,3) cycle in test_multigrid_gpu.py
TOL = {"f64": 2e-11, "f32": 4e-5}


@pytest.mark.parametrize("kind", ["f64", "f32"])
@pytest.mark.parametrize("nu", [(0, 3), (1, 2), (2, 3), (3, 0), (0, 1)])
@pytest.mark.parametrize("dim,k,L", [(2, 2, 3), (2, 3, 5), (3, 1, 3)])
def test_sweep_counts(cuda, dim, k, L, nu, kind):
    coarse = unit_square_mesh(k, 0.15, 0) if dim == 2 else unit_cube_kuhn_mesh(k, 0.1, 0)
    got, ref = _two_cycles(coarse, L, *nu, kind)
    np.testing.assert_allclose(got, ref, rtol=0, atol=TOL[kind] * np.abs(ref).max())


@pytest.mark.parametrize("kind", ["f64", "f32"])
@pytest.mark.parametrize("k,L", [(1, 6), (5, 3), (9, 2), (24, 2), (24, 0)])
def test_coarse_meshes(cuda, k, L, kind):
    got, ref = _two_cycles(unit_square_mesh(k, 0.15, 0), L, 3, 3, kind)
    np.testing.assert_allclose(got, ref, rtol=0, atol=TOL[kind] * np.abs(ref).max())


@pytest.mark.parametrize("L,nu,k", [(2, (3, 3), 12), (4, (3, 3), 12), (2, (1, 2), 12), (4, (1, 2), 12), (2, (0, 2), 12),
                                    (4, (0, 2), 12), (2, (3, 3), 46)])
def test_same_bits_as_the_separate_launches(cuda, L, nu, k):
    """A mesh of 8 macros alone takes the coarse levels in one launch; in a group
    with one of 288 macros, too large for that, it takes the levels above 0 in
    launches of its own, with one of 4232 macros level 0 too."""
    import torch
    import paper_2305_15116_gb300 as H
    ms = [unit_square_mesh(q, 0.15, q) for q in (2, k)]
    Ms = [H.Mesh(m.coords, m.cells).refine(L).solver_setup(L, *nu) for m in ms]
    bs, us, los = [], [], []
    for i, M in enumerate(Ms):
        b = torch.empty(M.num_slots(L)[0], dtype=torch.float64, device="cuda")
        M.poisson_rhs(L, i, 0.1, b)
        bs.append(b), us.append(torch.zeros_like(b)), los.append(torch.zeros_like(b))
    H.solve_two_part_group(Ms, L, bs, us, los, mode=H.SOLVE_MIXED, rtol=1e-9, max_iter=60)
    u, lo = torch.zeros_like(bs[0]), torch.zeros_like(bs[0])
    Ms[0].solve_two_part(L, bs[0], u, lo, mode=H.SOLVE_MIXED, rtol=1e-9, max_iter=60)
    assert torch.equal(u, us[0]) and torch.equal(lo, los[0])
    assert torch.isfinite(u).all() and u.abs().max() > 0
    for M in Ms:
        M.close()
