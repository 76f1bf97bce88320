"""3D products on fine levels, every slot: float-float, fp32 and native fp64 of
the same fp32-valued vector against each other, and the partial rows of a macro
alone against its products (needs a GPU)."""
import ctypes

import numpy as np
import pytest

from inputs import unit_cube_kuhn_mesh
import oracle

pytestmark = pytest.mark.gpu


def _macros(count):
    c = unit_cube_kuhn_mesh(1, 0.1, 4)
    used, cells = np.unique(c.cells[:count], return_inverse=True)
    return c.coords[used] + 0.05 * np.random.default_rng(7).standard_normal((len(used), 3)), cells.reshape(-1, 4)


@pytest.mark.parametrize("L,count", [(7, 1), (8, 1), (8, 3), (8, 6), (9, 1), (9, 2), (10, 1), (11, 1)])
def test_every_slot(cuda, L, count):
    import torch
    import paper_2305_15116_gb300 as H
    from paper_2305_15116_gb300 import _capi as C
    coords, cells = _macros(count)
    M = H.Mesh(coords, cells, bc=H.BC_NONE).refine(L)
    ns, ng = M.num_slots(L)
    g = torch.Generator(device="cuda").manual_seed(L)
    x = torch.rand(ng if count > 1 else ns, generator=g, device="cuda") * 2 - 1
    if count > 1:
        x = x[torch.from_numpy(M.dof_map(L)).cuda()]
    # the largest row sum of |a_ij|: all kinds of rows occur on level 2, whose
    # weights are 2^(L-2) times those of level L
    A = oracle.operator_matrix(oracle.RefinedMesh(coords, cells, 2, dirichlet=False))
    R = abs(A).sum(axis=1).max() * 2.0 ** (2 - L)
    xd = x.double()
    y = torch.full_like(xd, float("nan"))
    M.apply(L, xd, y, ieee=True)
    y64 = torch.full_like(xd, float("nan"))
    M.apply(L, xd, y64)
    # 1e-13 of sum |a_ij x_j| for float-float; native: a product and at most 15
    # fused terms per copy and 24 copies, each an ulp of 2^-53
    err = (y64 - y).abs_().max().item()
    assert err <= (1e-13 + 40 * 2.0 ** -53) * R, err
    y32 = torch.full_like(x, float("nan"))
    M.apply(L, x, y32)
    y.sub_(y32)
    err = y.abs_().max().item()
    assert err <= 41 * 2.0 ** -24 * R, err  # the same chain in fp32 and the rounded weights
    if count == 1:  # one macro: its partial rows are its products
        for code, v, want in ((H.F64, xd, y64), (H.F32, x, y32)):
            p = torch.full_like(v, float("nan"))
            C.check(C.lib.hyteg_apply_partial(M._h, L, code, v.data_ptr(), p.data_ptr(),
                                              ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "partial")
            assert torch.equal(p, want)
    M.close()


@pytest.mark.parametrize("odd", [0.0, 1e-4])
@pytest.mark.parametrize("kind,L,count", [("f64_ieee", 8, 2), ("f64_ieee", 8, 4), ("f64", 7, 6), ("f32", 7, 6),
                                          ("f64", 7, 3), ("f32", 7, 3), ("f64", 8, 2)])
def test_a_macro_alone_has_the_same_bits(cuda, kind, L, count, odd):
    """Marched (native fp64 on level 8, six macros on level 7) or walked along rows in
    a mesh, a macro's partial rows are those of the macro alone, which takes rows or a
    thread per point."""
    import torch
    import paper_2305_15116_gb300 as H
    from paper_2305_15116_gb300 import _capi as C
    coords, cells = _macros(count)
    code = {"f64": H.F64, "f32": H.F32, "f64_ieee": H.F64_IEEE}[kind]

    def partial(M, x):
        y = torch.full_like(x, float("nan"))
        C.check(C.lib.hyteg_apply_partial(M._h, L, code, x.data_ptr(), y.data_ptr(),
                                          ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "partial")
        return y
    M = H.Mesh(coords, cells, bc=H.BC_NONE).refine(L)
    ns, _ = M.num_slots(L)
    S = ns // count
    g = torch.Generator(device="cuda").manual_seed(count)
    x = torch.rand(ns, generator=g, device="cuda", dtype=torch.float64) * 2 - 1
    pick = torch.rand(ns, generator=g, device="cuda") < odd  # outside the float-float range, inside fp32's
    x = torch.where(pick, x * 1e-30, x).to(torch.float32 if kind == "f32" else torch.float64)
    y = partial(M, x)
    for c in (0, count - 1):
        One = H.Mesh(coords[cells[c]], np.arange(4)[None], bc=H.BC_NONE).refine(L)
        assert torch.equal(partial(One, x[c * S:(c + 1) * S].clone()), y[c * S:(c + 1) * S]), (kind, c)
        One.close()
    M.close()
