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


@pytest.mark.parametrize("count", [1, 2, 3, 6, 48])
def test_kernel_of_a_3d_level(count):
    """A thread per point for at most 2^20 slots (native fp64 up to level 7), rows for
    fine levels, the march between them."""
    out = fake_cuda.run(f"""
    m = unit_cube_kuhn_mesh(2, 0.1, 0)
    used, cells = np.unique(m.cells[:{count}], return_inverse=True)
    M = H.Mesh(m.coords[used], cells.reshape(-1, 4)).refine(9)
    for level in (5, 6, 7, 8, 9):
        r = []
        for dtype in (H.F64, H.F32, H.F64_IEEE):
            clear()
            assert apply(M, level, dtype) == 0
            l, = launches()
            r.append([k for k in ("Direct3", "March3", "Rows3") if k in l["name"]][0][0])
        print("".join(r))
    """)
    march6, march7 = count >= 22, count >= 6
    seven = "DDD" if count <= 2 else "MMD" if march7 else "RRD"
    assert out == ["MMD" if count >= 162 else "DDD", "MMD" if march6 else "DDD", seven,
                   "RRR" if count % 2 else "RRM", "RRR"]


def test_fused_sweeps_of_fine_3d_levels():
    out = fake_cuda.run("""
    M = H.Mesh(np.eye(4)[:, :3], np.arange(4)[None]).refine(8).solver_setup(8)
    clear()
    print(C.lib.hyteg_vcycle(M._h, 8, H.F32, X, Y, None), sum("Rows3" in l["name"] for l in launches()),
          any("Jacobi" in l["name"] for l in launches()))
    """)
    assert out == ["0 7 False"]


@pytest.mark.parametrize("k,level", [(1, 7), (2, 5), (5, 5), (8, 1), (32, 1), (45, 2)])
def test_coarse_levels_of_a_cycle(k, level):
    """The coarse levels' kernel takes the levels that give each of its 192 warps at
    most one task of a phase (level 0: 32 slots), the others are launches."""
    out = fake_cuda.run(f"""
    m = unit_square_mesh({k}, 0.1, 0)
    M = H.Mesh(m.coords, m.cells).refine({level}).solver_setup({level})
    clear()
    assert C.lib.hyteg_vcycle(M._h, {level}, H.F32, X, Y, None) == 0
    coarse = [l["cluster"] for l in launches() if "k_coarse" in l["name"]]
    top, cells = -1, len(m.cells)
    V, E = ({k} + 1) ** 2, 3 * {k} ** 2 + 2 * {k}
    for l in range({level} + 1):
        n = 2 ** l
        tasks = (3 * cells + 31) // 32 if l == 0 else V + E * ((n - 1 + 31) // 32) + cells * (((n - 1) * (n - 2) // 2 + 31) // 32)
        if tasks > 192:
            break
        top = l
    # a launch per phase above: two more pre-sweeps (three on the finest level), the
    # residual, both transfers, three sweeps; the level-0 solve where it is a launch
    n = sum(8 + (l == {level}) for l in range(1, {level} + 1) if l > top) + 1
    print(coarse == ([16] if top >= 0 else []), len(launches()) == n, top)
    """)
    assert out[0].startswith("True True"), out


@pytest.mark.parametrize("k", [1, 3])
def test_no_second_round_in_the_coarse_levels(k):
    out = fake_cuda.run(f"""
    m = unit_square_mesh(24, 0.1, 0)
    M = H.Mesh(m.coords, m.cells).refine({k}).solver_setup({k})
    clear()
    C.lib.hyteg_vcycle(M._h, {k}, H.F32, X, Y, None)
    print(len(launches()) > 8 * {k})
    """)
    assert out == ["True"]


def test_no_tiles_for_levels_that_are_not_walked():
    """A 2D level whose products take a thread per point is refined without the
    walker's two tile lists."""
    out = fake_cuda.run("""
    from inputs import rect_mesh
    m = rect_mesh(3, 1, 0.1, 0)
    M = H.Mesh(m.coords, m.cells).refine(7)
    n = []
    for level in (8, 9):  # 199 k and 791 k slots
        a = F.fake_uploads()
        M.refine(level)
        n.append(F.fake_uploads() - a)
        clear()
        apply(M, level)
        n.append("Direct2" in launches()[0]["name"])
    print(n[2] - n[0], n[1], n[3])
    """)
    assert out == ["2 True False"]
