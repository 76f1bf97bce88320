"""3D apply on macro-tets around one axis: edges and vertices with more copies
than other meshes have (40 on an axis edge, 80 on the centre vertex: more than
a warp has lanes), faces of two copies and Dirichlet points, on levels with
and without points inside edges, faces and macros; against the oracle, and the
partial apply's copies summed against the apply (needs a GPU)."""
import numpy as np
import pytest

from parity import oracle_reference, check_close, gpu_apply

pytestmark = pytest.mark.gpu


def _fan(k):
    """k tets around each half of the axis a - c - b, jittered ring."""
    rng = np.random.default_rng(5)
    ang = 2 * np.pi * np.arange(k) / k
    ring = np.stack([np.cos(ang), np.sin(ang), 0.1 * rng.uniform(-1, 1, k)], axis=1)
    coords = np.concatenate([[[0, 0, 1.0], [0.02, -0.03, 0.05], [0, 0, -1.1]], ring])
    cells = []
    for i in range(k):
        p, q = 3 + i, 3 + (i + 1) % k
        cells += [(0, 1, p, q), (1, q, 2, p)]

    class C:
        pass
    C.coords, C.cells = coords, np.array(cells, dtype=np.int64)
    return C


@pytest.mark.parametrize("kind", ["f64", "f32", "f64_ieee"])
@pytest.mark.parametrize("k,L", [(5, 3), (13, 2), (40, 0), (40, 1), (40, 3)])
@pytest.mark.parametrize("bc", [True, False])
def test_fan_of_tets(cuda, kind, k, L, bc):
    import torch
    import paper_2305_15116_gb300 as H
    from paper_2305_15116_gb300 import _capi as C
    import ctypes
    c = _fan(k)
    M = H.Mesh(c.coords, c.cells, bc=H.BC_DIRICHLET if bc else H.BC_NONE).refine(L)
    rm, x, y, absrow = oracle_reference(c, L, bc=bc, x_seed=3, kind=kind)
    smap = M.dof_map(L)
    yg = gpu_apply(M, L, x[smap], kind)
    check_close(yg, y[smap], absrow[smap], kind, f"fan {k} L{L}")
    # the partial rows of the copies add up, in ascending macro order, to the row
    dt = torch.float32 if kind == "f32" else torch.float64
    code = {"f32": H.F32, "f64": H.F64, "f64_ieee": H.F64_IEEE}[kind]
    xs = torch.from_numpy(x[smap]).to("cuda", dt)
    part = torch.full_like(xs, float("nan"))
    C.check(C.lib.hyteg_apply_partial(M._h, L, code, ctypes.c_void_p(xs.data_ptr()), ctypes.c_void_p(part.data_ptr()),
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "partial")
    torch.cuda.synchronize()
    part = part.cpu().numpy()
    total = np.zeros(rm.n_global, dtype=part.dtype)
    for s, g in enumerate(smap):
        total[g] = total[g] + part[s]
    free = ~M.dirichlet_mask(L)
    got = total[smap].astype(np.float64)
    assert np.array_equal(got[free], yg[free])
    M.close()
