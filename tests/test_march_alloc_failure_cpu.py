"""3D products on a level during whose refinement an allocation failed: the level
marches over its macros like one that was refined undisturbed (the library on a
CUDA runtime without a GPU, fake_cudart.cpp)."""
import fake_cuda


def test_no_product_without_its_macros():
    out = fake_cuda.run("""
    m = unit_cube_kuhn_mesh(3, 0.1, 0)
    def mesh(n):
        used, cells = np.unique(m.cells[:n], return_inverse=True)
        return H.Mesh(m.coords[used], cells.reshape(-1, 4))
    def grids(M):
        out = []
        for dtype in (H.F64, H.F32, H.F64_IEEE):
            clear()
            out.append((apply(M, 6, dtype), [l["grid"] for l in launches()]))
        return out
    refused = kept = 0
    for k in range(100):
        n = 22 + k  # from 2^20 slots on, a number of macros that is tuned for the first time
        M = mesh(n).refine(5)
        F.fake_fail_malloc(k, 0)  # the allocation k of level 6
        r = C.lib.hyteg_mesh_refine(M._h, 6)
        armed = F.fake_malloc_armed()
        F.fake_fail_malloc(-1, 0)
        if armed:
            break
        assert r in (0, -2), r  # HYTEG_ENOMEM
        if r:
            assert C.lib.hyteg_mesh_refine(M._h, 6) == 0
        refused, kept = refused + (r != 0), kept + (r == 0)
        fresh = mesh(n).refine(6)
        assert grids(M) == grids(fresh), (k, r, grids(M), grids(fresh))
        M.close(), fresh.close()
    print(refused > 5, kept > 5, armed)
    """)
    assert out == ["True True 1"]
