"""Small systems are cleared by a kernel that the tile kernels overlap: every entry is written, call after call, on a
side stream and in a captured graph, whatever A and b held before; odd sizes and the persistent launch too."""
import pytest

from paper_1805_03949_gb300 import meshgen as mg
from tests.helpers import FP32_TOL, FP64_TOL, engine, err_vs_oracle

pytestmark = pytest.mark.gpu

MESHES = {"mixed": lambda: mg.hybrid_cube(6, 3), "hex": lambda: mg.hex_cube(0, 0.2, 5, nx=3, ny=4, nz=5),
          "one": lambda: mg.hex_cube(1)}


@pytest.mark.parametrize("schedule", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("name", list(MESHES))
def test_overlapped_clearing(oracle, name, kind, precision, schedule):
    import torch
    fea = engine()
    mesh = MESHES[name]()
    ref = oracle.assemble(mesh, kind)
    s = fea.System.from_mesh(mesh, 1 if kind == 0 else 3)
    tol = FP64_TOL if precision == 0 else FP32_TOL

    def check():
        errA, zA = err_vs_oracle(s.A.cpu().numpy(), ref["A"], ref["NA"])
        errb, zb = err_vs_oracle(s.b.cpu().numpy(), ref["b"], ref["Nb"])
        assert max(errA, zA, errb, zb) <= tol, (errA, zA, errb, zb)

    try:
        op = fea.make_operator(kind=kind, precision=precision, schedule=schedule)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            for _ in range(20):
                s.A.fill_(float("nan"))
                s.b.fill_(float("nan"))
                s.assemble(op)
                s.assemble(op)
        side.synchronize()
        check()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            s.assemble(op)
        for _ in range(3):
            s.A.fill_(float("nan"))
            s.b.fill_(float("nan"))
            graph.replay()
        torch.cuda.synchronize()
        check()
        s.check()
    finally:
        s.close()
