"""Tile kernels that start while their system is still being cleared: each of many rounds and graph replays gives the
oracle's system, whatever A and b held, with few CTAs, some hundred light ones and more than a thousand; the
elastoplastic tiles, which write the new state before they wait, too."""
import numpy as np
import pytest

from paper_1805_03949_gb300 import meshgen as mg
from tests.helpers import FP32_TOL, FP64_TOL, engine, err_vs_oracle

pytestmark = pytest.mark.gpu

# name: mesh, kind; tets: 32 per CTA, and A stays below 32 MB
CASES = {"mixed_j2": (lambda: mg.hybrid_cube(5, 3), 2), "mixed_finite_strain": (lambda: mg.hybrid_cube(5, 3), 3),
         "hex_j2": (lambda: mg.hex_cube(6, 0.2, 2), 2),
         "tets_324_ctas": (lambda: mg.template_cube(12, mg.TET4, 0.2, 8), 0),
         "tets_1094_ctas": (lambda: mg.template_cube(18, mg.TET4, 0.2, 8), 0),
         "tets_1094_ctas_elasticity": (lambda: mg.template_cube(18, mg.TET4, 0.2, 8), 1)}
# two runs differ by the order of the additions alone: at most 2 n 2^-53 of the largest entry for the n <= 48 elements
# of an entry
ORDER = 96 * 2.0 ** -53


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_every_round_is_whole(oracle, name, precision):
    import torch
    fea = engine()
    factory, kind = CASES[name]
    mesh = factory()
    s = fea.System.from_mesh(mesh, 1 if kind == 0 else 3)
    assert s.A.numel() * 8 <= 32 << 20
    kw, state = {}, None
    if kind >= 2:
        U = mg.fourier_displacement(mesh.coords, 1.5e-4 if kind == 2 else 0.004, seed=4)
        kw["u"] = torch.tensor(U.reshape(-1), device="cuda")
        ref = oracle.j2_assemble(mesh, U) if kind == 2 else oracle.nh_assemble(mesh, U)
        if kind == 2:
            state = kw["state_out"] = torch.zeros((mesh.n_elems, 8, 7), dtype=torch.float64, device="cuda")
    else:
        ref = oracle.assemble(mesh, kind)
    try:
        op = fea.make_operator(kind=kind, precision=precision, **kw)
        s.assemble(op)
        s.check()
        tol = FP64_TOL if precision == 0 else FP32_TOL
        errs = err_vs_oracle(s.A.cpu().numpy(), ref["A"], ref["NA"]) + err_vs_oracle(s.b.cpu().numpy(), ref["b"], ref["Nb"])
        assert max(errs) <= tol, errs
        A0, b0, st0 = s.A.clone(), s.b.clone(), None if state is None else state.clone()
        worst = torch.zeros(3, dtype=torch.float64, device="cuda")
        graph = torch.cuda.CUDAGraph()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            with torch.cuda.graph(graph, stream=side):
                s.assemble(op, stream=side)
            for k in range(60):
                s.A.fill_(float("nan"))
                s.b.fill_(float("nan"))
                if state is not None:
                    state.fill_(float("nan"))
                if k % 3 == 2:
                    graph.replay()
                else:
                    s.assemble(op, stream=side)
                    if k % 3:
                        s.assemble(op, stream=side)
                worst[0] = torch.maximum(worst[0], (s.A - A0).abs().max())   # a NaN stays
                worst[1] = torch.maximum(worst[1], (s.b - b0).abs().max())
                if state is not None:
                    same = (state == st0) | (state.isnan() & (st0 == 0))     # slots past an element's points are not written
                    worst[2] = torch.maximum(worst[2], (~same).sum().double())
        side.synchronize()
        s.check()
        got = worst.cpu().numpy()
        assert got[0] <= ORDER * float(A0.abs().max()) and got[1] <= ORDER * max(float(b0.abs().max()), 1e-300), got
        assert got[2] == 0 and np.isfinite(got).all(), got
    finally:
        s.close()
