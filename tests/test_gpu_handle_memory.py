"""Device memory of a mesh handle: a mesh of one element type keeps its coordinates, offsets, types and connectivity, and
no lists per type; a mesh of several types keeps those too."""
import numpy as np
import pytest

from paper_1805_03949_gb300 import meshgen as mg
from tests.helpers import engine

pytestmark = pytest.mark.gpu

SLACK = 6 << 20   # two allocations rounded up to the driver's 2 MB pages, and small arrays


@pytest.mark.parametrize("mixed", [False, True])
def test_upload_keeps_what_is_read(mixed):
    import torch
    fea = engine()
    mesh = mg.hex_cube(80, 0.0, 1)
    if mixed:   # a tet after the hexes, on their first nodes
        tet = np.array([0, 1, 81, 81 * 81], dtype=mesh.conn.dtype)
        mesh = mg.Mesh(mesh.coords, np.append(mesh.types, np.uint8(mg.TET4)),
                       np.append(mesh.conn_offsets, mesh.conn_offsets[-1] + 4), np.append(mesh.conn, tet))
    N, E, L = len(mesh.coords), mesh.n_elems, len(mesh.conn)
    torch.cuda.synchronize()
    fea.fea_mesh_destroy(fea.fea_mesh_upload(mg.hex_cube(1).coords, *_arrays(mg.hex_cube(1))))   # the context is up
    free = torch.cuda.mem_get_info()[0]
    h = fea.fea_mesh_upload(mesh.coords, *_arrays(mesh))
    try:
        used = free - torch.cuda.mem_get_info()[0]
    finally:
        fea.fea_mesh_destroy(h)
    need = 24 * N + 17 * E + 4 * L + (12 * E + 4 * L if mixed else 0)
    assert need - SLACK <= used <= need + SLACK, (used, need)


def _arrays(mesh):
    return mesh.types, mesh.conn_offsets, mesh.conn
