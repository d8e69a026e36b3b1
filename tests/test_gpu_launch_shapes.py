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
