"""Pattern, map and upload where their kernels change path: nodes of many elements, element counts around a
tile, host and device input, and inputs that are refused."""
import numpy as np
import pytest

from paper_1805_03949_gb300 import meshgen as mg
from tests.helpers import engine

pytestmark = pytest.mark.gpu


def _fan(k):
    """k tetrahedra around the edge of nodes 0 and 1 (both ends lie in all of them)."""
    a = 2 * np.pi * np.arange(k) / k
    ring = np.stack([np.cos(a), np.sin(a), np.full(k, 0.5)], axis=1)
    coords = np.concatenate([[[0.0, 0.0, 0.0], [0.0, 0.0, 1.0]], ring])
    i = np.arange(k)
    conn = np.stack([np.zeros(k), 2 + i, 2 + (i + 1) % k, np.ones(k)], axis=1).astype(np.int32)
    return mg.Mesh(coords, np.full(k, mg.TET4, np.uint8), 4 * np.arange(k + 1, dtype=np.int64), conn.reshape(-1))


def _on(mesh, where):
    if where == "host":
        return mesh
    import torch
    return mg.Mesh(*(torch.tensor(v, device="cuda") for v in (mesh.coords, mesh.types, mesh.conn_offsets, mesh.conn)))


def _check(fea, oracle, mesh, where, ndof):
    n = mesh.n_elems
    s = fea.System.from_mesh(_on(mesh, where), ndof)
    try:
        assert s.n_elems == n
        rp, col, nmap = oracle.pattern(mesh, ndof)
        assert np.array_equal(s.row_ptr.cpu().numpy(), rp)
        assert np.array_equal(s.col_idx.cpu().numpy(), col)
        assert np.array_equal(s.node_map.cpu().numpy(), nmap)
        t, f, c = fea.fea_work_items(s.handle, 7)
        assert [int(c[t == k].sum()) for k in range(4)] == [int((mesh.types == k).sum()) for k in range(4)]
    finally:
        s.close()


@pytest.mark.parametrize("k", [3, 63, 64, 65, 127, 129, 256])
def test_nodes_of_many_elements(oracle, k):
    _check(engine(), oracle, _fan(k), "device", 3)


def test_too_many_elements_around_a_node_are_refused():
    fea = engine()
    with pytest.raises(fea.FeaError) as e:
        fea.System.from_mesh(_fan(257), 1)
    assert e.value.code == fea.FEA_ERR_UNSUPPORTED


@pytest.mark.parametrize("where", ["host", "device"])
@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 2100])
def test_mixed_upload_around_a_tile(oracle, n, where):
    mesh = mg.hybrid_cube(8, 5)
    at = mesh.conn_offsets[n]
    _check(engine(), oracle, mg.Mesh(mesh.coords, mesh.types[:n], mesh.conn_offsets[:n + 1], mesh.conn[:at]), where, 1)


@pytest.mark.parametrize("where", ["host", "device"])
def test_refused_input_names_the_first_fault(where):
    fea = engine()
    good = mg.hybrid_cube(6, 5)

    def message(**change):
        a = dict(types=good.types.copy(), conn_offsets=good.conn_offsets.copy(), conn=good.conn.copy())
        for name, edits in change.items():
            for at, value in edits:
                a[name][at] = value
        with pytest.raises(fea.FeaError) as e:
            fea.System.from_mesh(_on(mg.Mesh(good.coords, **a), where), 1)
        assert e.value.code == fea.FEA_ERR_ARG
        return str(e.value)

    E = good.n_elems
    assert "conn_offsets[0] != 0" in message(conn_offsets=[(0, 1)])
    assert "unknown element type at element 5" in message(types=[(900, 7), (5, 4)])
    assert f"does not match the node count of element {E - 1}" in message(conn_offsets=[(E, 2 ** 40)])
    assert "does not match the node count of element 3" in message(conn_offsets=[(4, 1)], types=[(900, 9)])
    assert "node id out of range at conn[17]" in message(conn=[(40, good.n_nodes), (17, -1)])
