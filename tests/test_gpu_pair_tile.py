"""The FP64 pair tiles at the edges of a tile: element counts around the tile size, every type and race treatment."""
import pytest

from paper_1805_03949_gb300 import meshgen as mg
from tests.helpers import FP64_TOL, engine, err_vs_oracle

pytestmark = pytest.mark.gpu

# elements per tile (PairCfg::EPC of pair_tile.cuh)
TILE = {mg.TET4: 32, mg.PYR5: 16, mg.PRISM6: 20, mg.HEX8: 16}
# scatter, schedule: atomic, coloring, multidependences, work stealing
PATHS = [(0, 0), (1, 0), (4, 0), (0, 1)]


@pytest.mark.parametrize("extra", [None, -1, 0, 1])
@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("etype", list(TILE))
def test_pair_tile_edges(oracle, etype, kind, extra):
    fea = engine()
    n = 1 if extra is None else 2 * TILE[etype] + extra
    mesh = mg.template_cube(3, etype, 0.2, 9)
    nn = mg.NODES_PER_TYPE[etype]
    mesh = mg.Mesh(mesh.coords, mesh.types[:n], mesh.conn_offsets[:n + 1], mesh.conn[:n * nn])
    assert mesh.n_elems == n
    params = dict(k0=0.5, k2=2.0, source=1.5) if kind == 0 else dict(young=2.0, poisson=0.2)
    ref = oracle.assemble(mesh, kind, **params)
    s = fea.System.from_mesh(mesh, 1 if kind == 0 else 3)
    try:
        for scatter, schedule in PATHS:
            s.A.fill_(float("nan"))
            s.assemble(fea.make_operator(kind=kind, precision=0, scatter=scatter, schedule=schedule, chunk=24, **params))
            s.check()
            errA, zA = err_vs_oracle(s.A.cpu().numpy(), ref["A"], ref["NA"])
            errb, zb = err_vs_oracle(s.b.cpu().numpy(), ref["b"], ref["Nb"])
            assert max(errA, zA, errb, zb) <= FP64_TOL, (scatter, schedule, errA, zA, errb, zb)
    finally:
        s.close()
