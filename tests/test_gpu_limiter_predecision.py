"""The limiter's l = 1 test is pre-decided on FP32 values and pairs of them: over
states whose neighbours differ by anything from a few ulps to order one, and
for gamma on and off the 7/5 path, the first pass's limiter must be the
oracle's, entry by entry, but for roundoff decisions. Needs a GPU."""
import numpy as np
import pytest

import oracle
from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M
from paper_2106_02159_gb300 import workloads as W

from . import test_gpu_parity_limiter as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [1.4, 1.3, 5.0 / 3.0])
@pytest.mark.parametrize("kind", ["q1", "hex"])
def test_limiter_decisions_are_the_oracles(kind, gamma, monkeypatch):
    B.build()
    monkeypatch.setattr(L, "GAMMA", gamma)
    if kind == "q1":
        mesh = M.structured_q1(30, 17, 0.0, 2.0, 0.0, 1.0, periodic_y=True)
    else:
        mesh = M.structured_q1_3d(8, 6, 5, kinds=(M.BC_SLIP,) * 6)
    rng = np.random.default_rng(5)
    noise = rng.uniform(-1.0, 1.0, (4, mesh.n))
    hat = np.exp(-((mesh.coords - mesh.coords.mean(0)) ** 2).sum(1) / 0.1)
    one = np.ones(mesh.n)
    zero = [0.0 * one] * (mesh.dim - 1)
    states = [(f"noise {a:g}", W.conserved(1.4 * (1.0 + a * noise[0]), [3.0 + a * noise[1]] + zero, 1.0 + a * noise[2],
                                           gamma)) for a in (1e-15, 1e-13, 1e-11, 1e-9, 1e-7, 1e-5, 1e-3, 0.3)]
    states.append(("isentropic", W.conserved(1.0 + 0.5 * hat, [1.0 * one] + zero, (1.0 + 0.5 * hat) ** gamma, gamma)))
    # densities and energies outside the FP32 powers' ranges
    states.append(("light", W.conserved(1e-4 * (1.0 + hat), [one] + zero, 1e-3 * (1.0 + hat), gamma)))
    states.append(("dense", W.conserved(1e4 * (1.0 + hat), [one] + zero, 1e9 * (1.0 + hat * hat), gamma)))
    orc = oracle.Oracle(mesh, gamma=gamma)
    s = B.Solver(dim=mesh.dim, gamma=gamma)
    s.upload_mesh(mesh)
    for name, U in states:
        _, tau, tr = orc.forward_euler(U, trace=True)
        s.set_state(U)
        s.stage(tau)
        l_gpu, l_orc = s.trace(B.EH_TRACE_L_PASS1), tr["lij"][0]
        bad = L.illegitimate_flips(mesh, L.limiter_flips(l_gpu, l_orc), l_gpu, l_orc, tr["UL"], tr["P"], tr["bounds"])
        assert bad.size == 0, (name, bad.size, l_gpu[bad[:4]], l_orc[bad[:4]])
