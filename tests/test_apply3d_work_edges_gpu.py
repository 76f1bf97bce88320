"""The edges of the 3D march's work on a tuned level against the oracle's rows:
the first and last slices of every z-range (equal slice counts) and the first and
last columns of every block of 256 (needs a GPU)."""
import numpy as np
import pytest

from inputs import unit_cube_kuhn_mesh, random_vector
import oracle
from parity import check_close, gpu_apply
from test_apply_2d_gpu import _absrow

pytestmark = pytest.mark.gpu


def _row(t):  # the row of point t of a triangle with rows of 1, 2, 3, .. points
    j = int((np.sqrt(8.0 * t + 1.0) - 1.0) / 2.0)
    return j - 1 if j * (j + 1) // 2 > t else j + 1 if (j + 1) * (j + 2) // 2 <= t else j


def _edge_points(n, chunks, dense):
    """Macro-interior points (x, y, z) of the slices next to a cut, in columns on
    both sides of a block's end; a column is a point counted from a slice's end."""
    cuts = [(n + 1) * c // chunks for c in range(chunks + 1)]
    pts = set()
    for z0, z1 in zip(cuts, cuts[1:]):
        zlo = max(1, z0)
        kmax = n - 1 - zlo
        first, end = (0, kmax * (kmax - 1) // 2) if dense else (3, (kmax + 1) * (kmax + 2) // 2)
        for b in range(first, end + 256, 256):
            for t in (b - 1, b):
                if not first <= t < end:
                    continue
                k = _row(t) + 2 if dense else _row(t)
                j = 1 + t - (k - 2) * (k - 1) // 2 if dense else t - k * (k + 1) // 2
                for z in {zlo, (zlo + z1) // 2, z1 - 1}:
                    x, y = k - j, n - z - k
                    if x >= 1 and y >= 1 and z >= 1 and x + y + z < n:
                        pts.add((x, y, z))
    return sorted(pts)


@pytest.mark.parametrize("kind", ["f64", "f32"])
def test_tuned_level(cuda, kind):
    import paper_2305_15116_gb300 as H
    coarse, L = unit_cube_kuhn_mesh(2, 0.1, 5), 6
    M = H.Mesh(coarse.coords, coarse.cells).refine(L)
    chunks = M.autotune_choice(L, H.F32 if kind == "f32" else H.F64)
    assert chunks > 0
    n = 1 << L
    ns, ng = M.num_slots(L)
    S = ns // coarse.n_cells
    smap = M.dof_map(L)
    x = random_vector(ng, 9)
    if kind == "f32":
        x = x.astype(np.float32).astype(np.float64)
    yg = gpu_apply(M, L, x[smap], kind)
    N = n + 1
    pts = _edge_points(n, chunks, kind == "f64")
    assert len(pts) > 20
    slot = [N * (N + 1) * (N + 2) // 6 - (N - z) * (N - z + 1) * (N - z + 2) // 6 + py * (N - z) - py * (py - 1) // 2 + px
            for px, py, z in pts]
    slots = np.concatenate([np.array(slot) + c * S for c in (0, 1, 22, coarse.n_cells - 1)])
    rm = oracle.RefinedMesh(coarse.coords, coarse.cells, L)
    gids = smap[slots]
    absrow = np.array([_absrow(rm, g, x) for g in gids])
    check_close(yg[slots], oracle.row_apply(rm, gids, x), absrow, kind, f"edges of {chunks} z-ranges")
    M.close()
