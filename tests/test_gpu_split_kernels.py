"""Small meshes run the split forms of the row kernels (a 32-row chunk per block,
its entries or components dealt out to warps) and few queued line searches run
by lane pairs; large meshes run a thread per row. An instance of a large batch
must therefore equal the same mesh alone, bit for bit, for every row length,
number of limiter passes and precision. Needs a GPU."""
import numpy as np
import pytest

from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M
from paper_2106_02159_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ROWS = 70_000  # above every bound of the split forms


def _fan(spokes):
    """P1 triangles around one node: a row of spokes + 1 entries (> 64: the
    limiter's long-row path), the others of 4."""
    a = 2.0 * np.pi * np.arange(spokes) / spokes
    coords = np.concatenate([[[0.0, 0.0]], np.stack([np.cos(a), np.sin(a)], -1)])
    r = np.arange(spokes)
    cells = np.stack([np.zeros(spokes, dtype=np.int64), 1 + r, 1 + (r + 1) % spokes], 1)
    faces = np.stack([1 + r, 1 + (r + 1) % spokes], 1)
    return M._finish(f"fan{spokes}", 2, coords, cells, coords[cells], M._local_p1, faces, coords[faces],
                     np.full(spokes, M.BC_DO_NOTHING), r)


MESHES = {
    "p1": lambda: M.periodic_p1_square(13),
    "q1": lambda: M.cylinder_channel_q1(7),
    "fan": lambda: _fan(90),
    "hex": lambda: M.structured_q1_3d(5, 4, 6, kinds=(M.BC_SLIP,) * 6),
}


@pytest.mark.parametrize("kind,passes,precision,gamma", [
    ("p1", 2, B.EH_PRECISION_FP64, 1.4), ("q1", 2, B.EH_PRECISION_FP64, 1.4), ("q1", 3, B.EH_PRECISION_MIXED, 1.4),
    ("q1", 1, B.EH_PRECISION_FP64, 1.3), ("fan", 2, B.EH_PRECISION_FP64, 1.4), ("fan", 3, B.EH_PRECISION_MIXED, 1.3),
    ("hex", 2, B.EH_PRECISION_FP64, 1.4), ("hex", 2, B.EH_PRECISION_MIXED, 1.4)])
def test_split_forms_equal_the_row_forms(kind, passes, precision, gamma):
    B.build()
    mesh = MESHES[kind]()
    copies = ROWS // mesh.n + 1
    base = dict(rho=1.4, vel=(3.0, 0.2), p=1.0)
    variety = [W.perturbed_state(mesh, k, base=base, amplitude=0.1 * (k % 4), gamma=gamma) for k in range(8)]
    bs1 = np.ascontiguousarray(W.uniform_state(mesh, gamma=gamma)[:, mesh.bnd_node])
    big, off, bs = M.concatenate([mesh] * copies, [bs1] * copies)
    kw = dict(dim=mesh.dim, gamma=gamma, limiter_passes=passes, precision=precision)
    s = B.Solver(**kw)
    s.upload_mesh(big, bs)
    s.set_instances(off)
    s.set_state(np.concatenate([variety[k % 8] for k in range(copies)], axis=1))
    s.run(3)
    U = s.get_state()
    searches = 0
    for k in range(8):
        one = B.Solver(**kw)
        one.upload_mesh(mesh, bs1)
        one.set_state(variety[k])
        one.run(3)
        searches += one.diagnostics()["line_searches_iterated"]
        assert np.array_equal(one.get_state(), U[:, off[k]:off[k + 1]]), (kind, k)
    assert searches > 0 or kind == "fan"  # the lane pairs ran
    d = s.diagnostics()
    assert d["not_admissible"] == 0 and d["line_searches_iterated"] >= searches
