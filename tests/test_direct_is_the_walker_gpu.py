"""The direct kernels (small vectors) and the walkers (large ones) give the same
bits, also where single inputs lie outside the float-float range and their rows
are recomputed in native fp64: one macro alone (direct) against the same macro
in a mesh that is walked (2D) or marched (3D) (needs a GPU)."""
import ctypes

import numpy as np
import pytest

from inputs import unit_square_mesh, unit_cube_kuhn_mesh

pytestmark = pytest.mark.gpu


def _partial(M, L, code, x):
    import torch
    from paper_2305_15116_gb300 import _capi as C
    y = torch.full_like(x, float("nan"))
    C.check(C.lib.hyteg_apply_partial(M._h, L, code, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()),
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "partial")
    torch.cuda.synchronize()
    return y


@pytest.mark.parametrize("kind", ["f64", "f32", "f64_ieee"])
@pytest.mark.parametrize("odd", [0.0, 1e-3])
@pytest.mark.parametrize("dim,k,L", [(2, 5, 7), (2, 3, 9), (3, 2, 6)])
def test_same_bits(cuda, kind, odd, dim, k, L):
    import torch
    import paper_2305_15116_gb300 as H
    coarse = unit_square_mesh(k, 0.15, 1) if dim == 2 else unit_cube_kuhn_mesh(k, 0.1, 1)
    dt = torch.float32 if kind == "f32" else torch.float64
    code = {"f64": H.F64, "f32": H.F32, "f64_ieee": H.F64_IEEE}[kind]
    M = H.Mesh(coarse.coords, coarse.cells, bc=H.BC_NONE).refine(L)
    ns, _ = M.num_slots(L)
    S = ns // coarse.n_cells
    rng = np.random.default_rng(8)
    v = rng.uniform(-1, 1, ns)
    pick = rng.random(ns) < odd
    v[pick] *= rng.choice([1e-30, 1e25], pick.sum())  # outside the float-float range, inside fp32's
    x = torch.from_numpy(v).to("cuda", dt)
    y = _partial(M, L, code, x)
    for c in (0, coarse.n_cells - 1):
        One = H.Mesh(coarse.coords[coarse.cells[c]], np.arange(dim + 1)[None], bc=H.BC_NONE).refine(L)
        assert torch.equal(_partial(One, L, code, x[c * S:(c + 1) * S].clone()), y[c * S:(c + 1) * S]), (kind, c)
        One.close()
    M.close()
