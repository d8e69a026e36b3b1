"""eh_cfl_dt_noalloc does not check c_ij: a pattern may hold entries with c_ij = 0,
whose d_ij is 0 whether the two states are equal or not. Needs a GPU."""
import numpy as np
import pytest

from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M
from paper_2106_02159_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("amplitude", [0.0, 0.2])
@pytest.mark.parametrize("dim", [2, 3])
def test_entries_without_coupling(dim, amplitude):
    torch = pytest.importorskip("torch")
    mesh = M.cylinder_channel_q1(20) if dim == 2 else M.structured_q1_3d(6, 5, 7, kinds=(M.BC_SLIP,) * 6)
    U = W.perturbed_state(mesh, 2, amplitude=amplitude)
    rows, col = mesh.row_of_entry(), mesh.col
    cij = mesh.cij.copy()
    cij[:, (rows != col) & ((rows + col) % 7 == 0)] = 0.0  # both directions of an edge
    # the method's sum over the entries that couple, in plain FP64
    gamma, boundary = 1.4, np.zeros(mesh.n, dtype=bool)
    boundary[mesh.bnd_node] = True
    rho, vel = U[0], U[1:1 + dim] / U[0]
    p = (gamma - 1.0) * (U[-1] - 0.5 * rho * (vel * vel).sum(0))
    a = np.sqrt(gamma * p / rho)
    az = a * p ** (-(gamma - 1.0) / (2.0 * gamma))
    norm = np.sqrt((cij * cij).sum(0))
    some = (rows != col) & (norm > 0.0)
    k = np.nonzero(some)[0]

    def bound(left, right, entry):
        n = cij[:, entry] / norm[entry]
        ul, ur = (vel[:, left] * n).sum(0), (vel[:, right] * n).sum(0)
        x = np.maximum(a[left] + a[right] - 0.5 * (gamma - 1.0) * (ur - ul), 0.0) / (az[left] + az[right])
        ps = x ** (2.0 * gamma / (gamma - 1.0))
        s = [np.sqrt(1.0 + (gamma + 1.0) / (2.0 * gamma) * np.maximum(ps / p[q] - 1.0, 0.0)) for q in (left, right)]
        return np.maximum(np.maximum(a[left] * s[0] - ul, ur + a[right] * s[1]), 0.0) * norm[entry]

    order = np.full(mesh.nnz, -1)
    order[np.lexsort((rows, col))] = np.arange(mesh.nnz)  # the transposed entry of a symmetric pattern
    up = np.where(rows < col, np.arange(mesh.nnz), order)[k]
    lo, hi = np.minimum(rows, col)[k], np.maximum(rows, col)[k]
    d = bound(lo, hi, up)
    d = np.where(boundary[lo] & boundary[hi], np.maximum(d, bound(hi, lo, order[up])), d)
    total = np.bincount(rows[k], weights=d, minlength=mesh.n)
    expect = (0.5 * mesh.mi[total > 0] / (2.0 * total[total > 0])).min()
    dev = lambda x, t: torch.as_tensor(np.ascontiguousarray(x, dtype=t), device="cuda")  # noqa: E731
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    B.cfl_dt_noalloc(dim, gamma, 0.5, dev(mesh.row_ptr, np.int64), dev(col, np.int32), dev(cij, np.float64),
                     dev(mesh.mi, np.float64), dev(boundary, np.uint8), dev(U, np.float64), out)
    assert abs(float(out.item()) - expect) <= 1e-12 * expect, (float(out.item()), expect)
