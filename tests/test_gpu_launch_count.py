"""fea_assemble_launches against the kernels that one captured fea_assemble call holds: every operator, scatter and
schedule, on systems cleared by a kernel and by memsets."""
import ctypes

import pytest

from paper_1805_03949_gb300 import meshgen as mg
from tests.helpers import engine

pytestmark = pytest.mark.gpu

MESHES = {"small_mixed": lambda: mg.hybrid_cube(5, 3), "small_hex": lambda: mg.hex_cube(5, 0.2, 2),
          "large_hex": lambda: mg.hex_cube(27, 0.2, 2)}   # A of 3 dofs per node: 0.4, 0.1 and 41 MB
SCATTERS = {"atomic": 0, "color": 1, "rows": 2, "block": 3, "multidep": 4}


def captured_kernels(torch, call):
    """Kernel nodes of the CUDA graph that `call` enqueues (nothing runs)."""
    cu = ctypes.CDLL("libcuda.so.1")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph, n = ctypes.c_void_p(), ctypes.c_size_t()
    h = ctypes.c_void_p(stream.cuda_stream)
    assert cu.cuStreamBeginCapture_v2(h, 1) == 0          # CU_STREAM_CAPTURE_MODE_THREAD_LOCAL
    try:
        call(stream)
    finally:
        assert cu.cuStreamEndCapture(h, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kernels = 0
    for node in nodes:
        kind = ctypes.c_int()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kernels += kind.value == 0                        # CU_GRAPH_NODE_TYPE_KERNEL
    assert cu.cuGraphDestroy(graph) == 0
    return kernels


@pytest.mark.parametrize("kind", [0, 1, 2, 3])
@pytest.mark.parametrize("name", list(MESHES))
def test_count_is_what_a_call_launches(name, kind):
    import torch
    fea = engine()
    mesh = MESHES[name]()
    s = fea.System.from_mesh(mesh, 1 if kind == 0 else 3)
    kw = dict(kind=kind)
    if kind >= 2:
        kw["u"] = torch.tensor(mg.fourier_displacement(mesh.coords, 1e-4, seed=4).reshape(-1), device="cuda")
    solid = kind in (2, 3)
    paths = [(sc, 0) for sc in SCATTERS if not solid or sc in ("atomic", "color")]
    paths += [("atomic", sch) for sch in (1, 2, 3) if kind != 3]
    try:
        for precision in (0, 1):
            for scatter, schedule in paths:
                args = dict(kw, precision=precision, scatter=SCATTERS[scatter], schedule=schedule)
                if schedule > 1:
                    n = len(fea.fea_work_items(s.handle, 0)[0])
                    args.update(queue=torch.arange(n, dtype=torch.int32, device="cuda"), n_ctas=1,
                                queue_off=torch.tensor([0, n], dtype=torch.int64, device="cuda"))
                op = fea.make_operator(**args)
                s.assemble(op)                            # the first call builds the plans
                s.check()
                want = captured_kernels(torch, lambda stream: s.assemble(op, stream=stream))
                got = fea.fea_assemble_launches(op, s.handle)
                assert got == want, (scatter, schedule, precision, got, want)
        s.check()
    finally:
        s.close()


def test_bench_events_end_with_the_tile():
    """The benchmark's events of an atomic or colored step: as many as tile launches, whatever clears the system."""
    import bench
    fea = engine()
    s = {k: fea.System.from_mesh(MESHES[k](), 3) for k in ("small_hex", "large_hex")}
    try:
        post = {}
        for key, system in s.items():
            for name, op in bench.variant_operators(fea).items():
                system.assemble(op)
                launches = fea.fea_assemble_launches(op, system.handle)
                post[key, name] = bench.kernels_after_zeroing(fea, system, name, launches)
                assert 0 <= launches - post[key, name] <= 1
            system.check()
        for key, system in s.items():
            colors = fea.fea_color_info(system.handle, system.n_elems)[0]
            assert post[key, "fp64_atomic"] == post[key, "fp32_atomic"] == 1 and post[key, "fp32_color"] == colors
            assert post[key, "fp32_block"] == 1
    finally:
        for system in s.values():
            system.close()
