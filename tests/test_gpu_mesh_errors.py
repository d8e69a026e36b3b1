"""What eh_upload_mesh says of a bad mesh: the first error in the order of the
checks (rows, pattern, coefficients, boundary list) with its row and column, the
same one every time whichever kernel thread finds one first, and EH_ERR_BAD_MESH
also where the device has no room for the mesh. Needs a GPU."""
import dataclasses

import numpy as np
import pytest

from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M

pytestmark = pytest.mark.gpu


def _mesh():
    return M.cylinder_channel_q1(40)


def _refusal(s, mesh, bs):
    with pytest.raises(B.EulerError) as e:
        s.upload_mesh(mesh, bs)
    assert e.value.status == B.EH_ERR_BAD_MESH, str(e.value)
    return str(e.value)


def _with(mesh, **changes):
    """The mesh with single values of its arrays replaced: name = {index: value}."""
    out = {}
    for name, values in changes.items():
        out[name] = getattr(mesh, name).copy()
        for k, v in values.items():
            out[name][k] = v
    return dataclasses.replace(mesh, **out)


def _entry(mesh, row):
    """The last off-diagonal entry of a row and its column."""
    k = int(mesh.row_ptr[row + 1]) - 1
    k -= mesh.col[k] == row
    return k, int(mesh.col[k])


def _asymmetric(mesh, row):
    """Row `row` with its largest column replaced by one that it is not coupled
    to (the rows in between stay as they are)."""
    k0, k1 = int(mesh.row_ptr[row]), int(mesh.row_ptr[row + 1])
    new = next(c for c in range(mesh.n - 1, int(mesh.col[k1 - 1]), -1))
    assert new not in mesh.col[k0:k1] and mesh.col[k1 - 1] != row
    return k1 - 1, new


def test_messages_name_the_first_error():
    mesh = _mesh()
    bs = np.ones((4, mesh.n_bnd))
    s = B.Solver()
    lo, hi = mesh.n // 3, mesh.n - 200  # in different blocks of every kernel
    (kl, jl), (kh, jh) = _entry(mesh, lo), _entry(mesh, hi)
    two = lambda name, a, b, value: _with(mesh, **{name: {a: value, b: value}})  # noqa: E731
    k0 = int(mesh.row_ptr[lo])
    cases = [
        (two("col", kl, kh, mesh.n), f"column out of range in row {lo}"),
        (two("mi", lo, hi, 0.0), f"m_{lo} <= 0"),
        (two("mij", kl, kh, 7.0), f"consistent mass not symmetric at ({min(lo, jl)},{max(lo, jl)})"),
        (_with(mesh, col={k0 + 1: mesh.col[k0]}, mi={lo - 1: -1.0}), f"m_{lo - 1} <= 0"),
        (_with(mesh, col={k0 + 1: mesh.col[k0]}, mi={lo: -1.0}), f"row {lo} not sorted/unique"),
        (_with(mesh, cij={(slice(None), kl): 0.0}), "c_ij = 0 at an off-diagonal entry"),
        # an earlier check's error comes first, whatever its row
        (_with(mesh, cij={(slice(None), kl): 0.0}, col={kh: mesh.n}), f"column out of range in row {hi}"),
        (_with(mesh, row_ptr={hi + 1: mesh.row_ptr[hi]}, mi={lo: 0.0}), f"m_{lo} <= 0"),
        (_with(mesh, row_ptr={hi + 1: mesh.row_ptr[hi]}), f"row {hi} has fewer than 2 entries"),
        (_with(mesh, bnd_node={1: mesh.bnd_node[0]}), f"boundary node {mesh.bnd_node[0]} invalid or repeated"),
        (_with(mesh, bnd_node={1: mesh.bnd_node[0]}, mi={hi: 0.0}), f"m_{hi} <= 0"),
    ]
    for bad, text in cases:
        message = _refusal(s, bad, bs)
        assert f": {text} (status" in message, (message, text)
    s.upload_mesh(mesh, bs)


def test_the_first_of_many_asymmetric_rows_is_named():
    """Every second row with a column that does not point back: the first one is
    named with that column, every time."""
    mesh = _mesh()
    bs = np.ones((4, mesh.n_bnd))
    first = mesh.n // 4
    col = mesh.col.copy()
    names = {}
    for row in range(first, mesh.n - 400, 2):
        k, new = _asymmetric(mesh, row)
        names[row] = new
        col[k] = new
    bad = dataclasses.replace(mesh, col=col)
    # a row before the first one whose entry (i, j) lost its (j, i) is named instead
    rows = mesh.row_of_entry()
    pairs = set(zip(rows.tolist(), col.tolist()))
    i, j = next((i, j) for i, j in zip(rows.tolist(), col.tolist()) if (j, i) not in pairs)
    s = B.Solver()
    for _ in range(5):
        assert f": pattern not symmetric at ({i},{j}) (status" in _refusal(s, bad, bs)


@pytest.mark.parametrize("precision", [B.EH_PRECISION_FP64, B.EH_PRECISION_MIXED])
def test_a_bad_mesh_without_room(precision):
    torch = pytest.importorskip("torch")
    mesh = M.cylinder_channel_q1(225)
    bs = np.ones((4, mesh.n_bnd))
    s = B.Solver(precision=precision)
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    held = torch.empty(free - (128 << 20), dtype=torch.uint8, device="cuda")
    try:
        k, _ = _entry(mesh, mesh.n // 2)
        message = _refusal(s, _with(mesh, col={k: mesh.n}), bs)
        assert f": column out of range in row {mesh.n // 2} (status" in message
        with pytest.raises(B.EulerError) as e:
            s.upload_mesh(mesh, bs)
        assert e.value.status == B.EH_ERR_OOM
    finally:
        del held
        torch.cuda.empty_cache()
    s.upload_mesh(mesh, bs)
