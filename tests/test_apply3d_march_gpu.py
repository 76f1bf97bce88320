"""The 3D column march (large vectors) where it can go wrong: against the
direct kernel, macro by macro, on a mesh with an odd number of macros (the last
pair holds one) and vectors at odd element offsets, and against the oracle's
rows at a level whose slices need the larger ring (needs a GPU)."""
import ctypes

import numpy as np
import pytest

from inputs import unit_cube_kuhn_mesh, random_vector
import oracle
from parity import check_close, gpu_apply
from test_apply_2d_gpu import _absrow

pytestmark = pytest.mark.gpu

KINDS = ["f64", "f32", "f64_ieee"]


def _partial(M, L, code, x, y):
    import torch
    from paper_2305_15116_gb300 import _capi as C
    C.check(C.lib.hyteg_apply_partial(M._h, L, code, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()),
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "partial")
    return y


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("offset", [0, 1])
def test_march_is_bitwise_the_direct_kernel(cuda, kind, offset):
    import torch
    import paper_2305_15116_gb300 as H
    L = 6
    coarse = unit_cube_kuhn_mesh(2, 0.1, 3)
    used, cells = np.unique(coarse.cells[:25], return_inverse=True)  # 1.2M slots: marched
    coords, cells = coarse.coords[used], cells.reshape(25, 4)
    dt = torch.float32 if kind == "f32" else torch.float64
    code = {"f64": H.F64, "f32": H.F32, "f64_ieee": H.F64_IEEE}[kind]
    M = H.Mesh(coords, cells, bc=H.BC_NONE).refine(L)
    ns, _ = M.num_slots(L)
    assert ns >= 2 ** 20
    S = ns // 25
    g = torch.Generator().manual_seed(4)
    buf = (torch.rand(ns + 1, generator=g, dtype=torch.float64) * 2 - 1).to("cuda", dt)
    x = buf[offset:offset + ns]
    y = torch.full((ns + 1,), float("nan"), dtype=dt, device="cuda")[offset:offset + ns]
    _partial(M, L, code, x, y)
    for c in (0, 1, 11, 24):  # one macro alone: 48k slots, the direct kernel
        One = H.Mesh(coords[cells[c]], np.arange(4)[None], bc=H.BC_NONE).refine(L)
        xs = x[c * S:(c + 1) * S].clone()
        ys = _partial(One, L, code, xs, torch.full_like(xs, float("nan")))
        torch.cuda.synchronize()
        assert torch.equal(ys, y[c * S:(c + 1) * S]), (kind, c)
        One.close()
    M.close()


@pytest.mark.parametrize("kind", KINDS)
def test_level8_rows(cuda, kind):
    import paper_2305_15116_gb300 as H
    coarse, L = unit_cube_kuhn_mesh(1, 0.1, 4), 8
    M = H.Mesh(coarse.coords, coarse.cells).refine(L)
    ns, ng = M.num_slots(L)
    smap = M.dof_map(L)
    x = random_vector(ng, 6)
    if kind == "f32":
        x = x.astype(np.float32).astype(np.float64)
    yg = gpu_apply(M, L, x[smap], kind)
    assert np.all(np.isfinite(yg))
    rm = oracle.RefinedMesh(coarse.coords, coarse.cells, L)
    slots = np.random.default_rng(17).integers(0, ns, 300)
    gids = smap[slots]
    yref = oracle.row_apply(rm, gids, x)
    absrow = np.array([_absrow(rm, g, x) for g in gids])
    check_close(yg[slots], yref, absrow, kind, "3D L8 sampled")
    M.close()
