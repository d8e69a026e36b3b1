"""eh_cfl_dt_noalloc evaluates in FP64 only the rows that its FP32 brackets
leave as candidates for the smallest bound: the step must be the context's
(eh_cfl_dt evaluates every row) for states that make the brackets wide, tie
or fall out of FP32's range. Needs a GPU."""
import numpy as np
import pytest

from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M
from paper_2106_02159_gb300 import workloads as W

pytestmark = pytest.mark.gpu

DT_TOL = 1e-13  # the relative tolerance of the CFL step in the parity tests


def _states(mesh, gamma):
    rng = np.random.default_rng(11)
    one = np.ones(mesh.n)
    zero = [0.0 * one] * (mesh.dim - 1)
    x = mesh.coords
    hat = np.exp(-((x - x.mean(0)) ** 2).sum(1) / 0.05)
    noise = rng.uniform(-1.0, 1.0, (4, mesh.n))
    yield "uniform", W.conserved(1.4 * one, [3.0 * one] + zero, one, gamma)
    yield "at rest", W.conserved(one, [0.0 * one] + zero, one, gamma)
    # every row within the brackets' width of the smallest bound
    yield "ties", W.conserved(1.4 * (1.0 + 1e-9 * noise[0]), [3.0 * one] + zero, one, gamma)
    yield "rough", W.conserved(np.exp(noise[0]), [2.0 * noise[1]] + zero, np.exp(2.0 * noise[2]), gamma)
    yield "fast", W.conserved(one, [200.0 + hat] + zero, one + hat, gamma)
    yield "colliding", W.conserved(one, [-5.0 * np.tanh(50.0 * (x[:, 0] - x[:, 0].mean()))] + zero, 0.01 * one, gamma)
    yield "near vacuum", W.conserved(1e-6 + hat, [4.0 * np.tanh(50.0 * (x[:, 0] - x[:, 0].mean()))] + zero,
                                     1e-7 + hat, gamma)
    yield "tiny units", W.conserved(1e-40 * (1.0 + hat), [1e-9 * noise[1]] + zero, 1e-50 * (1.0 + hat), gamma)
    yield "large units", W.conserved(1e38 * (1.0 + hat), [1e9 * noise[1]] + zero, 1e55 * (1.0 + hat), gamma)


@pytest.mark.parametrize("gamma", [1.4, 1.05, 1.001, 5.0 / 3.0])
@pytest.mark.parametrize("kind", ["q1", "p1", "hex", "flat"])
def test_bracketed_step_is_the_contexts(kind, gamma):
    torch = pytest.importorskip("torch")
    B.build()
    mesh = {"q1": lambda: W.cylinder_problem(20)[0], "p1": lambda: M.periodic_p1_square(23),
            "hex": lambda: M.structured_q1_3d(6, 5, 7, kinds=(M.BC_SLIP,) * 6),
            "flat": lambda: M.structured_q1(130, 3, 0.0, 130.0, 0.0, 1e-3)}[kind]()
    bs = np.ascontiguousarray(W.uniform_state(mesh, gamma=gamma)[:, mesh.bnd_node])
    s = B.Solver(dim=mesh.dim, gamma=gamma, cfl=0.5)
    s.upload_mesh(mesh, bs)
    dev = lambda a, t: torch.as_tensor(np.ascontiguousarray(a, dtype=t), device="cuda")  # noqa: E731
    isb = np.zeros(mesh.n, dtype=np.uint8)
    isb[mesh.bnd_node] = 1
    args = (dev(mesh.row_ptr, np.int64), dev(mesh.col, np.int32), dev(mesh.cij, np.float64), dev(mesh.mi, np.float64),
            dev(isb, np.uint8) if mesh.n_bnd else None)
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    for name, U in _states(mesh, gamma):
        s.set_state(U)
        expect = s.cfl_dt()
        B.cfl_dt_noalloc(mesh.dim, gamma, 0.5, *args, dev(U, np.float64), out)
        got = float(out.item())
        assert abs(got - expect) <= DT_TOL * expect, (name, got, expect)
