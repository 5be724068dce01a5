"""A work-stealing launch with few items starts one CTA per item (so that no SM gets several while others have none), in
assembly and in the element loop; with a fuller grid every CTA starts."""
import pytest

from paper_1805_03949_gb300 import meshgen as mg
from tests.helpers import FP32_TOL, FP64_TOL, engine, err_vs_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["hex", "mixed"])
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("n_ctas", [0, 40, 3])
def test_few_items_take_a_cta_each(oracle, name, kind, n_ctas):
    import torch
    fea = engine()
    mesh = mg.hex_cube(8, 0.2, 2) if name == "hex" else mg.hybrid_cube(8, 5)
    s = fea.System.from_mesh(mesh, 1 if kind == 0 else 3)
    try:
        n = len(fea.fea_work_items(s.handle, 0)[0])
        cta = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        kw = dict(kind=kind, schedule=fea.FEA_SCHED_STEAL, n_ctas=n_ctas, item_cta=cta)
        if kind == 2:
            U = mg.fourier_displacement(mesh.coords, 1.5e-4, seed=4)
            kw["u"] = torch.tensor(U.reshape(-1), device="cuda")
            ref = oracle.j2_assemble(mesh, U)
        else:
            ref = oracle.assemble(mesh, kind)
        for precision in (0, 1):
            op = fea.make_operator(precision=precision, **kw)
            grid = n_ctas or fea.fea_persistent_grid(op, s.handle)
            launched = grid if n > grid - grid // 4 else n
            for _ in range(3):
                s.A.fill_(float("nan"))
                cta.fill_(-1)
                s.assemble(op)
                s.check()
                got = cta.cpu().numpy()
                assert (got >= 0).all() and (got < launched).all(), (grid, got)
            tol = FP64_TOL if precision == 0 else FP32_TOL
            err = err_vs_oracle(s.A.cpu().numpy(), ref["A"], ref["NA"])
            assert max(err) <= tol, err
        if kind == 2:
            cta.fill_(-1)
            fea.fea_element_loop(op, s.handle)
            s.check()
            grid = n_ctas or fea.fea_element_loop_grid(op, s.handle)
            got = cta.cpu().numpy()
            assert (got >= 0).all() and (got < (grid if n > grid - grid // 4 else n)).all(), (grid, got)
    finally:
        s.close()
