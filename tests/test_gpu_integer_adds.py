"""Large meshes run part of the row kernels' additions on the integer units, small
ones run them on the FP64 pipe: every result must be the same, bit for bit, over
equal states, cancellation, components that are zero or far apart in magnitude,
and operands too small for the integer form (left to the FP64 pipe). An instance
of a large batch must therefore equal the same mesh alone. Needs a GPU."""
import numpy as np
import pytest

from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M
from paper_2106_02159_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ROWS = 100_000  # above the line of every such kernel


def _states(mesh, gamma):
    rng = np.random.default_rng(3)
    base = dict(rho=1.4, vel=(0.5, 0.0, 0.0)[:mesh.dim], p=1.0)
    uniform = W.perturbed_state(mesh, 0, base=base, amplitude=0.0, gamma=gamma)
    out = [uniform]
    for size in (1e-290, 1e-160, 1e-14, 1e-6):  # a transverse momentum beside none, beside much larger components
        U = uniform.copy()
        U[2] += size * rng.standard_normal(mesh.n) * (rng.random(mesh.n) < 0.5)
        out.append(U)
    U = uniform.copy()  # neighbours one or a few units in the last place apart
    U[0] *= 1.0 + 2.0**-52 * rng.integers(-3, 4, mesh.n)
    out.append(U)
    for scale in (1e-12, 1.0, 1e9):
        out.append(scale * W.perturbed_state(mesh, 1, base=base, amplitude=0.3, gamma=gamma))
    return out


@pytest.mark.parametrize("dim,precision,gamma", [
    (2, B.EH_PRECISION_FP64, 1.4), (2, B.EH_PRECISION_MIXED, 1.4), (2, B.EH_PRECISION_FP64, 1.3),
    (3, B.EH_PRECISION_FP64, 1.4), (3, B.EH_PRECISION_MIXED, 1.4)])
def test_large_meshes_equal_small_ones(dim, precision, gamma):
    B.build()
    mesh = M.cylinder_channel_q1(6) if dim == 2 else M.structured_q1_3d(5, 4, 6, kinds=(M.BC_SLIP,) * 6)
    states = _states(mesh, gamma)
    copies = ROWS // mesh.n + 1
    bs1 = np.ascontiguousarray(W.uniform_state(mesh, gamma=gamma)[:, mesh.bnd_node])
    big, off, bs = M.concatenate([mesh] * copies, [bs1] * copies)
    assert big.n >= ROWS
    kw = dict(dim=dim, gamma=gamma, precision=precision)
    s = B.Solver(**kw)
    s.upload_mesh(big, bs)
    s.set_instances(off)
    s.set_state(np.concatenate([states[k % len(states)] for k in range(copies)], axis=1))
    s.run(2)
    U = s.get_state()
    for k, U0 in enumerate(states):
        one = B.Solver(**kw)
        one.upload_mesh(mesh, bs1)
        one.set_state(U0)
        one.run(2)
        assert np.array_equal(one.get_state(), U[:, off[k]:off[k + 1]]), k
    assert s.diagnostics()["not_admissible"] == 0
