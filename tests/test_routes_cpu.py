"""Which kernels a call launches, and how large (the library on a CUDA runtime
without a GPU, fake_cudart.cpp)."""
import pytest

import fake_cuda


@pytest.mark.parametrize("k,level", [(40, 0), (40, 1), (16, 3), (8, 5)])
def test_p2_boundary_points_share_blocks(k, level):
    """Low levels of many macros: the threads of a P2 launch are at most twice its
    boundary points and the lanes of its row tiles (a warp for 30 columns)."""
    out = fake_cuda.run(f"""
    m = unit_square_mesh({k}, 0.1, 0)
    M = H.Mesh(m.coords, m.cells).refine({level})
    for dtype in (H.F64, H.F32, H.F64_IEEE):
        clear()
        C.lib.hyteg_p2_apply(M._h, {level}, dtype, X, Y, None)
        rows, = [l for l in launches() if "k_p2_rows" in l["name"]]
        n = 2 ** {level}
        tiles = sum((n - x0 + 63) // 64 for x0 in range(0, n, 30))
        points = 4 * n - 2 if n > 1 else 3
        print(rows["grid"] * rows["block"] <= 2 * len(m.cells) * (points + 32 * tiles) + 512)
    """)
    assert out == ["True"] * 3
