"""The bytes that admission counts (eh_estimate_device_bytes,
eh_estimate_request_bytes) against what eh_upload_mesh and an admitted request
take of the device's memory. Needs a GPU."""
import numpy as np
import pytest

from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M
from paper_2106_02159_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BLOCK = 2 << 20  # the device's memory is handed out in blocks of 2 MiB
ARRAYS = 45      # arrays of a context, at most


def _free():
    torch = pytest.importorskip("torch")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("precision", [B.EH_PRECISION_FP64, B.EH_PRECISION_MIXED])
@pytest.mark.parametrize("dim", [2, 3])
def test_estimates_are_what_is_allocated(dim, precision):
    mesh = M.cylinder_channel_q1(225) if dim == 2 else M.extruded_q1(M.cylinder_channel_q1(30), 20)
    U = W.uniform_state(mesh)
    bs = np.ascontiguousarray(U[:, mesh.bnd_node])
    s = B.Solver(dim=dim, precision=precision)
    before = _free()
    s.upload_mesh(mesh, bs)
    taken = before - _free()
    s.close()
    est = B.estimate_device_bytes(dim, precision, mesh.n, mesh.nnz)
    # 10 % of headroom, up to 3 % more where the rounding of an array's size is on the estimate's side
    assert taken - ARRAYS * BLOCK <= est <= 1.13 * taken + BLOCK, (taken, est)
    # a merged request before the batch is assembled: its own copy of the mesh and its state
    batch = B.Batch(8 << 30, dim=dim, precision=precision)
    before = _free()
    ticket = batch.admit(mesh, U, 1.0, bs)
    taken = before - _free()
    part = B.estimate_request_bytes(dim, precision, B.EH_BATCH_MERGED, mesh.n, mesh.nnz, mesh.n_bnd) - est
    assert ticket is not None
    assert taken - ARRAYS * BLOCK <= part <= 1.13 * taken + BLOCK, (taken, part)
    batch.close()
