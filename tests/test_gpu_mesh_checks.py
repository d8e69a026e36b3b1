"""The mesh checks and static arrays that eh_upload_mesh makes on the device:
every kind of bad mesh is refused with its status, whatever the place, and a
good one after it is taken; the transpose index is the oracle's definition.
Needs a GPU."""
import dataclasses

import numpy as np
import pytest

from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M

pytestmark = pytest.mark.gpu


def _mesh(kind):
    return M.cylinder_channel_q1(9) if kind == "2d" else M.structured_q1_3d(4, 3, 5, kinds=(M.BC_SLIP,) * 6)


def _offdiag(mesh, row):
    """Position of the last off-diagonal entry of a row."""
    k = int(mesh.row_ptr[row + 1]) - 1
    return k if mesh.col[k] != row else k - 1


def _drop(mesh, k):
    """The mesh without entry k (and with its transpose)."""
    row = int(np.searchsorted(mesh.row_ptr, k, side="right")) - 1
    keep = np.arange(mesh.nnz) != k
    rp = mesh.row_ptr.copy()
    rp[row + 1:] -= 1
    return dataclasses.replace(mesh, row_ptr=rp, col=mesh.col[keep], cij=np.ascontiguousarray(mesh.cij[:, keep]),
                               mij=mesh.mij[keep])


def _bad(mesh, what, row):
    k = _offdiag(mesh, row)
    k0, k1 = int(mesh.row_ptr[row]), int(mesh.row_ptr[row + 1])
    col, cij, mij, mi = mesh.col.copy(), mesh.cij.copy(), mesh.mij.copy(), mesh.mi.copy()
    if what == "column":
        col[k] = mesh.n
    elif what == "negative column":
        col[k0] = -1
    elif what == "order":
        col[k1 - 1] = col[k1 - 2]
    elif what == "diagonal":
        return _drop(mesh, k0 + int(np.nonzero(mesh.col[k0:k1] == row)[0][0]))
    elif what == "pattern":
        return _drop(mesh, k)
    elif what == "mass":
        mi[row] = 0.0
    elif what == "cij":
        cij[:, k] = 0.0
    elif what == "mij":
        mij[k] *= 1.0 + 1e-9
    elif what == "row_ptr":
        rp = mesh.row_ptr.copy()
        rp[row + 1] = rp[row]
        return dataclasses.replace(mesh, row_ptr=rp)
    return dataclasses.replace(mesh, col=col, cij=cij, mij=mij, mi=mi)


@pytest.mark.parametrize("kind,precision", [("2d", B.EH_PRECISION_FP64), ("3d", B.EH_PRECISION_MIXED)])
def test_bad_meshes_are_refused(kind, precision):
    mesh = _mesh(kind)
    bs = np.ones((mesh.dim + 2, mesh.n_bnd))
    s = B.Solver(dim=mesh.dim, precision=precision)
    for what in ("column", "negative column", "order", "diagonal", "pattern", "mass", "cij", "mij", "row_ptr"):
        for row in (0, mesh.n // 2, mesh.n - 1):
            with pytest.raises(B.EulerError) as e:
                s.upload_mesh(_bad(mesh, what, row), bs)
            assert e.value.status == B.EH_ERR_BAD_MESH, (what, row)
    s.upload_mesh(mesh, bs)
    row_ptr, col, tr = s.mesh_index()
    rows = mesh.row_of_entry()
    assert np.array_equal(row_ptr, mesh.row_ptr) and np.array_equal(col, mesh.col)
    assert np.array_equal(rows[tr], mesh.col) and np.array_equal(mesh.col[tr], rows)
