"""The FP32 pre-decisions at the ends of FP32's range: a change of units by powers
of two (lengths, densities, velocities) scales the method's quantities by powers
of two, so what the solver gives in one system of units it has to give in another,
however small the numbers are. Needs a GPU."""
import dataclasses

import numpy as np
import pytest

from paper_2106_02159_gb300 import binding as B
from paper_2106_02159_gb300 import meshes as M
from paper_2106_02159_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _units(mesh, U, length, density, velocity):
    """Mesh and state in units in which lengths, densities and velocities are so many times larger."""
    d = mesh.dim
    mesh = dataclasses.replace(mesh, cij=mesh.cij * length ** (d - 1), mij=mesh.mij * length**d, mi=mesh.mi * length**d)
    scale = np.array([1.0] + [velocity] * d + [velocity**2]) * density
    return mesh, np.ascontiguousarray(U * scale[:, None])


@pytest.mark.parametrize("length,density,velocity", [(1.0, 1.0, 1.0), (2.0**-50, 2.0**-30, 2.0**70),
                                                     (2.0**-60, 2.0**-20, 2.0**62)])
def test_cfl_step_below_the_fp32_range(length, density, velocity):
    """A mesh of several waves of blocks whose last part has the smallest bound:
    the step is that of the part alone (bounds of 1e-38 and less are not brushed
    aside by the FP32 comparison with the minimum so far)."""
    part = M.cylinder_channel_q1(20)
    copies = 150
    slow, fast = (W.perturbed_state(part, 1, base=dict(rho=1.4, vel=(v, 0.0), p=1.0), amplitude=0.1) for v in (0.5, 9.0))
    dt = []
    for states in ([fast], [slow] * (copies - 1) + [fast]):
        mesh, _, bs = M.concatenate([part] * len(states), [np.ones((4, part.n_bnd))] * len(states))
        mesh, U = _units(mesh, np.concatenate(states, axis=1), length, density, velocity)
        s = B.Solver()
        s.upload_mesh(mesh, bs)
        s.set_state(U)
        dt.append(s.cfl_dt())
        s.close()
    assert dt[0] == dt[1], dt


@pytest.mark.parametrize("nv,dim", [(24, 2), (270, 2), (0, 3)])  # (270: 72900 rows, the integer forms)
def test_viscosity_on_very_small_meshes(nv, dim):
    """Slow flow on meshes whose v.c_ij are below FP32's range: d_ij scales with
    |c_ij| to the last bit (no product with a velocity is taken for 0 where the
    FP32 intervals choose the outer wave)."""
    mesh = M.periodic_p1_square(nv) if dim == 2 else M.structured_q1_3d(9, 8, 10, periodic=(True, True, True))
    rng = np.random.default_rng(4)
    rho, p = 1.0 + 1e-5 * rng.random(mesh.n), (1.0 + 1e-5 * rng.random(mesh.n)) / 1.4
    vel = 2e-5 * rng.standard_normal((dim, mesh.n))
    U = np.concatenate([rho[None], rho * vel, (p / 0.4 + 0.5 * rho * (vel * vel).sum(0))[None]])
    c_scale = 2.0**-112  # |c_ij| about 1e-35
    d = []
    for length in (1.0, c_scale if dim == 2 else c_scale**0.5):
        m, V = _units(mesh, U, length, 1.0, 1.0)
        s = B.Solver(dim=dim)
        s.upload_mesh(m)
        s.set_state(V)
        s.stage()
        d.append(s.trace(B.EH_TRACE_D_IJ))
        s.close()
    assert np.array_equal(d[0] * c_scale, d[1]), np.max(np.abs(d[1] / c_scale / d[0] - 1.0))


@pytest.mark.parametrize("density,velocity", [(1.0, 1.0), (2.0**-90, 2.0**17), (2.0**-95, 2.0**20)])
@pytest.mark.parametrize("dim", [2, 3])
def test_allocation_free_cfl_step_of_thin_gases(dim, density, velocity):
    """Momenta of 1e-22, whose squares are below FP32's range (a gas of 1e-27 kg/m^3
    at 1e5 m/s): the brackets still hold the bounds, and the step is eh_cfl_dt's to
    the tolerance of the parity tests."""
    torch = pytest.importorskip("torch")
    mesh = M.cylinder_channel_q1(30) if dim == 2 else M.structured_q1_3d(9, 8, 10, kinds=(M.BC_SLIP,) * 6)
    dev = lambda a, t: torch.as_tensor(np.ascontiguousarray(a, dtype=t), device="cuda")  # noqa: E731
    isb = np.zeros(mesh.n, dtype=np.uint8)
    isb[mesh.bnd_node] = 1
    args = (dev(mesh.row_ptr, np.int64), dev(mesh.col, np.int32), dev(mesh.cij, np.float64), dev(mesh.mi, np.float64),
            dev(isb, np.uint8))
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    s = B.Solver(dim=dim)
    s.upload_mesh(mesh, np.ones((dim + 2, mesh.n_bnd)))
    for seed in range(6):
        _, U = _units(mesh, W.perturbed_state(mesh, seed), 1.0, density, velocity)
        s.set_state(U)
        expect = s.cfl_dt()
        B.cfl_dt_noalloc(dim, 1.4, 0.5, *args, dev(U, np.float64), out)
        assert abs(float(out.item()) - expect) <= 1e-13 * expect, (seed, float(out.item()), expect)
