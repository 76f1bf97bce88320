"""Meshes on two devices of one process: the kernels' attributes and the
autotuner's choices belong to a device (the library on a CUDA runtime without a
GPU, fake_cudart.cpp)."""
import pytest

import fake_cuda


@pytest.mark.parametrize("order", [(0, 1), (1, 0)])
def test_coarse_cycle_on_both(order):
    out = fake_cuda.run(f"""
    m = unit_square_mesh(2, 0.1, 0)
    for d in {order}:
        F.cudaSetDevice(d)
        M = H.Mesh(m.coords, m.cells).refine(5).solver_setup(5)
        clear()
        r = C.lib.hyteg_vcycle(M._h, 5, H.F32, X, Y, None)
        print(r, [(l["dev"], l["cluster"]) for l in launches() if "k_coarse" in l["name"]])
    """)
    assert out == [f"0 [({d}, 16)]" for d in order]


def test_march_on_both():
    out = fake_cuda.run("""
    m = unit_cube_kuhn_mesh(1, 0.1, 0)
    for d in (0, 1):
        F.cudaSetDevice(d)
        M = H.Mesh(m.coords, m.cells).refine(8)
        for level in (7, 8):
            for dtype in (H.F64, H.F32, H.F64_IEEE):
                clear()
                print(d, apply(M, level, dtype), len(launches()))
    """)
    assert out == [f"{d} 0 1" for d in (0, 1) for _ in range(6)]


@pytest.mark.parametrize("mesh,level,kernel", [("unit_square_mesh(8, 0.1, 0)", 7, "k_interior2d"),
                                               ("unit_cube_kuhn_mesh(2, 0.1, 0)", 6, "March3")])
def test_each_device_is_tuned_once(mesh, level, kernel):
    out = fake_cuda.run(f"""
    m = {mesh}
    for d in (0, 1, 0, 1):
        F.cudaSetDevice(d)
        clear()
        H.Mesh(m.coords, m.cells).refine({level})
        print(any("{kernel}" in l["name"] for l in launches()))
    """)
    assert out == ["True", "True", "False", "False"]
