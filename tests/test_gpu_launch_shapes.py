"""Launch shapes where they apply and where they do not: the row forms of the
kernels, FP64 and mixed, 2D and 3D, give the same bits for every block size and
with capped grids whose loops wrap; the autotuner leaves the shapes of kernels
that run in their split form as they are. Needs a GPU."""
import numpy as np
import pytest

from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M
from paper_2106_02159_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("passes", [2, 3])
def test_autotune_keeps_shapes_that_have_no_effect(passes):
    mesh, U0, bs = W.cylinder_problem(20)
    s = B.Solver(limiter_passes=passes)
    s.upload_mesh(mesh, bs)
    s.set_state(U0)
    s.apply_boundary_conditions()
    # (no candidate of the autotuner, so that none can be kept by chance)
    fixed = {"low": (128, 0), "lim1": (256, 333)} | ({"pass": (256, 333)} if passes == 2 else {})
    for kernel, shape in fixed.items():
        s.set_launch_shape(kernel, *shape)
    chosen = s.autotune(1)
    for kernel, (tpb, cap) in fixed.items():
        assert chosen[kernel] == s.block_sizes()[kernel] == tpb and s.rows_per_sm()[kernel] == cap, kernel
    if passes == 3:  # the second limiter pass is a row form: one of the candidates
        assert s.rows_per_sm()["pass"] in (0, 256, 512, 768)


def _copies(mesh, rows, kinds=8):
    """The mesh repeated to at least so many rows, with `kinds` states in turn:
    (big mesh, row offsets, boundary states, big state, states, boundary state)."""
    copies = rows // mesh.n + 1
    states = [W.perturbed_state(mesh, k, amplitude=0.1 * (1 + k % 4)) for k in range(kinds)]
    bs1 = np.ascontiguousarray(W.uniform_state(mesh)[:, mesh.bnd_node])
    big, off, bs = M.concatenate([mesh] * copies, [bs1] * copies)
    assert big.n >= rows
    return big, off, bs, np.concatenate([states[k % kinds] for k in range(copies)], axis=1), states, bs1


def _run(mesh, bs, off, U, steps, shape=None, **kw):
    s = B.Solver(dim=mesh.dim, **kw)
    s.upload_mesh(mesh, bs)
    if off is not None:
        s.set_instances(off)
    if shape is not None:
        tpb, cap = shape
        for kernel in ("lim1", "pass", "final"):
            s.set_launch_shape(kernel, tpb, cap)
        for kernel in ("prep", "visc", "low", "lsearch"):
            s.set_launch_shape(kernel, tpb)
    s.set_state(U)
    s.run(steps)
    out = s.get_state()
    d = s.diagnostics()
    s.close()
    return out, d


# above the last line at which a row kernel changes its form (k_low and k_lim1 add on
# the integer units from 98304 rows on); 152 SMs x 512 rows are fewer, so every cap wraps
ROW_FORMS = 100_000


@pytest.mark.parametrize("dim,precision,gamma", [
    (2, B.EH_PRECISION_FP64, 1.4), (2, B.EH_PRECISION_MIXED, 1.4), (2, B.EH_PRECISION_FP64, 1.3),
    (3, B.EH_PRECISION_FP64, 1.4), (3, B.EH_PRECISION_MIXED, 1.4)])
def test_row_forms_of_any_shape_give_the_same_bits(dim, precision, gamma):
    mesh = M.cylinder_channel_q1(16) if dim == 2 else M.structured_q1_3d(9, 8, 7, kinds=(M.BC_SLIP,) * 6)
    big, off, bs, U, _, _ = _copies(mesh, ROW_FORMS)
    kw = dict(precision=precision, gamma=gamma, limiter_passes=3)
    ref, d = _run(big, bs, off, U, 2, **kw)
    assert d["line_searches_deferred"] > 0 and d["not_admissible"] == 0
    for shape in ((64, 64), (128, 512), (256, 256), (256, 0)):
        out, q = _run(big, bs, off, U, 2, shape, **kw)
        assert np.array_equal(out, ref) and q["line_searches_deferred"] == d["line_searches_deferred"], shape


PAIRS = 608 * 32 // 2  # searches of a pass up to which lane pairs run them


@pytest.mark.parametrize("rows,precision", [  # k_visc: two warps a chunk of rows, and one
    (170_000, B.EH_PRECISION_FP64), (170_000, B.EH_PRECISION_MIXED),
    (660_000, B.EH_PRECISION_FP64), (660_000, B.EH_PRECISION_MIXED)])
def test_large_batches_equal_their_instances(rows, precision):
    """k_visc by two warps or one a chunk, and at gamma = 7/5 queues that a lane per
    search runs, against four warps and the lane pairs of the same mesh alone."""
    mesh = M.cylinder_channel_q1(16)
    big, off, bs, U, states, bs1 = _copies(mesh, rows)
    steps = 2
    out, d = _run(big, bs, off, U, steps, precision=precision)
    # 3 stages of 2 passes a step: one pass at least is above the pairs' line
    assert d["line_searches_deferred"] > steps * 6 * PAIRS
    for k, state in enumerate(states):
        one, e = _run(mesh, bs1, None, state, steps, precision=precision)
        assert 0 < e["line_searches_deferred"] <= steps * 6 * PAIRS
        assert np.array_equal(one, out[:, off[k]:off[k + 1]]), k
