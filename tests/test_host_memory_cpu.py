"""Host memory that runs out inside a C entry is HYTEG_ENOMEM, not an exception
thrown at the caller (the library on a CUDA runtime without a GPU,
fake_cudart.cpp, whose allocation k fails)."""
import pytest

import fake_cuda

MESHES = {2: "unit_square_mesh(2, 0.1, 0)", 3: "unit_cube_kuhn_mesh(1, 0.1, 0)"}
CALLS = {
    "apply": "apply(M, 5)",
    "partial": "C.lib.hyteg_apply_partial(M._h, 5, H.F64, X, Y, None)",
    "batch": "C.lib.hyteg_apply_batch(h, l, H.F64, x, y, 2, None)",
    "vcycle": "C.lib.hyteg_vcycle(M._h, 5, H.F32, X, Y, None)",
    "restrict": "C.lib.hyteg_restrict(M._h, 5, H.F32, X, Y, None)",
    "p2": "C.lib.hyteg_p2_apply(M._h, 5, H.F64, X, Y, None)",
}


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("call", sorted(CALLS))
def test_out_of_memory_is_a_status(dim, call):
    if dim == 3 and call == "p2":
        pytest.skip("P2 is two-dimensional")
    out = fake_cuda.run(f"""
    m = {MESHES[dim]}
    M = H.Mesh(m.coords, m.cells).refine(5).solver_setup(5)
    h, l = (ctypes.c_void_p * 2)(M._h, M._h), (ctypes.c_int * 2)(5, 4)
    x, y = (ctypes.c_void_p * 2)(X, X), (ctypes.c_void_p * 2)(Y, Y)
    codes = []
    for k in range(2000):
        F.fake_fail_new(k)
        r = {CALLS[call]}
        armed = F.fake_new_armed()
        F.fake_fail_new(-1)
        codes.append(r)
        if armed:
            break
    print(armed, codes[-1], set(codes[:-1]) <= {{-2}})
    """)
    assert out == ["1 0 True"]
