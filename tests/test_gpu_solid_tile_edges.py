"""Element tiles at the edges of a tile: element counts around the tile size for the elastoplastic and the finite-strain
solid in both precisions, the FP32 elasticity tiles, and the FP64 pyramids of diffusion and elasticity (32 per tile)."""
import numpy as np
import pytest

from paper_1805_03949_gb300 import meshgen as mg
from tests.helpers import FP32_TOL, FP64_TOL, engine, err_vs_oracle, j2_point_errors

pytestmark = pytest.mark.gpu

PAIR = {mg.TET4: 32, mg.PYR5: 16, mg.PRISM6: 20, mg.HEX8: 16}    # J2PairCfg, NHPairCfg (FP64)
ROWS = {mg.TET4: 32, mg.PYR5: 24, mg.PRISM6: 20, mg.HEX8: 16}    # J2Cfg, NHCfg, TileCfg (FP32)
POINTS = {mg.TET4: 4, mg.PYR5: 8, mg.PRISM6: 6, mg.HEX8: 8}


def _part(etype, n):
    """The first n elements of a jittered cube."""
    mesh = mg.template_cube(4, etype, 0.2, 9)
    nn = mg.NODES_PER_TYPE[etype]
    assert mesh.n_elems >= n
    return mg.Mesh(mesh.coords, mesh.types[:n], mesh.conn_offsets[:n + 1], mesh.conn[:n * nn])


def _counts(tile):
    return [1, tile - 1, tile, tile + 1, 2 * tile + 1]


def _check(s, ref, precision):
    tol = FP64_TOL if precision == 0 else FP32_TOL
    s.check()
    errA, zA = err_vs_oracle(s.A.cpu().numpy(), ref["A"], ref["NA"])
    errb, zb = err_vs_oracle(s.b.cpu().numpy(), ref["b"], ref["Nb"])
    assert max(errA, zA, errb, zb) <= tol, (errA, zA, errb, zb)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("etype", list(PAIR))
def test_j2_tile_edges(oracle, etype, precision):
    import torch
    fea = engine()
    for n in _counts((PAIR if precision == 0 else ROWS)[etype]):
        mesh = _part(etype, n)
        U = mg.fourier_displacement(mesh.coords, 1.5e-4, seed=4)
        ref, pts = oracle.j2_assemble(mesh, U), oracle.j2_points(mesh, U)
        mask = np.broadcast_to(np.arange(8) < POINTS[etype], (n, 8))
        s = fea.System.from_mesh(mesh, 3)
        try:
            u = torch.tensor(U.reshape(-1), device="cuda")
            for scatter, schedule in ((0, 0), (1, 0), (0, 1)):
                state = torch.full((n, 8, 7), float("nan"), dtype=torch.float64, device="cuda")
                s.A.fill_(float("nan"))
                s.assemble(fea.make_operator(kind=2, precision=precision, scatter=scatter, schedule=schedule, chunk=24,
                                             u=u, state_out=state))
                _check(s, ref, precision)
                err, _ = j2_point_errors(state.cpu().numpy(), None, ref["state"], pts["stress"], mask)
                assert err <= FP64_TOL, (n, scatter, schedule, err)
        finally:
            s.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("etype", list(PAIR))
def test_finite_strain_tile_edges(oracle, etype, precision):
    import torch
    fea = engine()
    for n in _counts((PAIR if precision == 0 else ROWS)[etype]):
        mesh = _part(etype, n)
        U = mg.fourier_displacement(mesh.coords, 0.004, seed=6) + 0.05 * mesh.coords[:, [1, 2, 0]]
        ref = oracle.nh_assemble(mesh, U, young=1.0, poisson=0.3, mass=0.5)
        s = fea.System.from_mesh(mesh, 3)
        try:
            u = torch.tensor(U.reshape(-1), device="cuda")
            for scatter in (0, 1):
                s.A.fill_(float("nan"))
                s.assemble(fea.make_operator(kind=3, precision=precision, scatter=scatter, u=u, young=1.0, poisson=0.3,
                                             mass=0.5))
                _check(s, ref, precision)
        finally:
            s.close()


@pytest.mark.parametrize("case", [(1, 1, t) for t in ROWS] + [(0, 0, mg.PYR5), (1, 0, mg.PYR5)])
def test_small_strain_tile_edges(oracle, case):
    fea = engine()
    kind, precision, etype = case
    for n in _counts(ROWS[etype] if precision else 32):
        mesh = _part(etype, n)
        params = dict(k0=0.5, k2=2.0, source=1.5) if kind == 0 else dict(young=2.0, poisson=0.2)
        ref = oracle.assemble(mesh, kind, **params)
        s = fea.System.from_mesh(mesh, 1 if kind == 0 else 3)
        try:
            for scatter, schedule in ((0, 0), (1, 0), (4, 0), (0, 1)):
                s.A.fill_(float("nan"))
                s.assemble(fea.make_operator(kind=kind, precision=precision, scatter=scatter, schedule=schedule,
                                             chunk=24, **params))
                _check(s, ref, precision)
        finally:
            s.close()
