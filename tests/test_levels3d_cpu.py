"""The range of levels of 3D products: up to 11, refused above with a message
that says so (the library on a CUDA runtime without a GPU, fake_cudart.cpp)."""
import fake_cuda


def test_level_12_is_refused_as_an_argument():
    out = fake_cuda.run("""
    M = H.Mesh(np.eye(4)[:, :3], np.arange(4)[None]).refine(12)
    for level in (11, 12):
        for dtype in (H.F64, H.F32, H.F64_IEEE):
            clear()
            h, l, x, y = (ctypes.c_void_p * 1)(M._h), (ctypes.c_int * 1)(level), (ctypes.c_void_p * 1)(X), (ctypes.c_void_p * 1)(Y)
            r = {apply(M, level, dtype), C.lib.hyteg_apply_partial(M._h, level, dtype, X, Y, None),
                 C.lib.hyteg_apply_batch(h, l, dtype, x, y, 1, None)}
            print(level, r, len(launches()), C.lib.hyteg_last_error().decode() if level > 11 else "")
    """)
    assert out == ["11 {0} 3 "] * 3 + ["12 {-1} 0 3D products take levels up to 11"] * 3


def test_native_fp64_marches_above_its_point_table_only():
    """Up to level 7 native products take the point table: there is no march kernel
    for them."""
    out = fake_cuda.run("""
    m = unit_cube_kuhn_mesh(2, 0.1, 0)
    M = H.Mesh(m.coords, m.cells).refine(5)
    marched = []
    for level in (6, 7, 8):
        M.refine(level)
        clear()
        apply(M, level, H.F64_IEEE)
        marched.append("March3" in launches()[0]["name"])
    print(marched, F.fake_has_kernel(b"March3INS_11ArF64Native", b"Li512E"))
    """)
    assert out == ["[False, False, True] 0"]
