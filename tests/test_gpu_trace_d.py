"""eh_trace(EH_TRACE_D_IJ): the symmetric d_ij and the diagonal -sum_j d_ij of the
last stage, in every layout of the edge data; reading it (with the search queue
as the scratch) leaves the following stages as they are. Needs a GPU."""
import numpy as np
import pytest

from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M
from paper_2106_02159_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [B.EH_PRECISION_FP64, B.EH_PRECISION_MIXED])
@pytest.mark.parametrize("kind,size", [("2d", 9), ("2d", 17), ("3d", 0)])  # 2d: below and above 8192 entries
def test_trace_of_d_between_stages(kind, size, precision):
    mesh = M.cylinder_channel_q1(size) if kind == "2d" else M.structured_q1_3d(5, 4, 6, kinds=(M.BC_SLIP,) * 6)
    U0 = W.perturbed_state(mesh, 5)
    bs = np.ascontiguousarray(W.uniform_state(mesh)[:, mesh.bnd_node])
    a, b = (B.Solver(dim=mesh.dim, precision=precision) for _ in range(2))
    for s in (a, b):
        s.upload_mesh(mesh, bs)
        s.set_state(U0)
    rows = mesh.row_of_entry()
    _, _, tr = a.mesh_index()
    off = rows != mesh.col
    for _ in range(3):
        a.stage()
        b.stage()
        d = a.trace(B.EH_TRACE_D_IJ)
        assert np.array_equal(d, a.trace(B.EH_TRACE_D_IJ))
        assert np.array_equal(d, d[tr]) and np.all(d[off] > 0)
        # the diagonal: the row's sum in FP64, stored in the precision of d (27 terms at most)
        eps = 27 * 2.0**-53 if precision == B.EH_PRECISION_FP64 else 2.0**-24
        total = np.bincount(rows[off], weights=d[off], minlength=mesh.n)
        assert np.all(np.abs(d[~off] + total) <= 1.01 * eps * total)
    assert np.array_equal(a.get_state(), b.get_state())
