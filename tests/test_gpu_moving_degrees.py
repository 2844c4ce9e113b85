"""Moving hexahedra of the highest degrees: their stage mass solves are
pointwise, so every N that a static mesh takes is taken by a moving one."""
import pytest

from gpu_util import TOL, rel_err, var_index
from test_gpu_moving import dg, setup, tgv  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [5, 6])
def test_moving_hexahedra(dg, N):  # noqa: F811
    box, vel, mo, mesh = setup(dg, "hex", 2, N)
    Q = tgv(mo)
    Qs = mesh.set_state(torch.from_numpy(Q).cuda())
    vidx = var_index(mo.mesh.nM)
    mesh.set_time(0.05)
    assert rel_err(mesh.get_state(mesh.rhs(Qs)), mo.rhs(Q, 0.05), vidx) < TOL
    dt = 1e-3
    mesh.set_time(0.0)
    mesh.rk_step(Qs, mesh.empty(), dt, 2)
    got, ref = mesh.get_state(Qs), mo.run(Q, 0.0, dt, 2)
    assert rel_err(got - Q, ref - Q, vidx) < 1e-10
    assert rel_err(got, ref, vidx) < TOL
    mesh.sync()
