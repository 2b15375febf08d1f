"""Every bead and every node counts once in the observables, at sizes where the
reductions' blocks take their second and third shares (more than 1,048,576
beads or nodes) and on both sides of that.

The velocities are eighths, whose squares and sums are exact, and the time step
is so small that the force leaves them alone: kinetic energy and momentum are
then known to the last bits of a float-float sum (2^-45 an addition, a few dozen
deep: 1e-12).  A bead left out or counted twice changes them by 1e-7 or more, a
node the field energy by as much.
"""
import numpy as np
import pytest

from paper_1310_2041_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FULL = 1 << 20


@pytest.mark.parametrize("n,mesh", [(FULL - 1, 101), (FULL, 102), (FULL + 1, 102), (2 * FULL + 513, 128),
                                    (3 * FULL - 257, 129)])
def test_observables_count_everything_once(hpf_gpu, n, mesh):
    w = W.Workload("free", [(n, [0])], float(mesh), mesh, 1, [[0.0]], 0.7, field_every=1, steps=1,
                   dt=1e-30, gamma=0.0)
    d = W.generate(w)
    rng = np.random.default_rng(n)
    vel = (rng.integers(8, 64, (n, 3)) / 8.0).astype(np.float32)
    with hpf_gpu.System(hpf_gpu.make_params(**w.params())) as s:
        s.set_state(d["pos"], vel, d["type"], d["bonds"])
        E = s.energy()
        D = s.scatter_density()
    assert E[0] == pytest.approx(0.5 * float((vel.astype(np.float64) ** 2).sum()), rel=1e-12)
    assert E[4] == pytest.approx(float(np.linalg.norm(vel.sum(0, dtype=np.float64))), rel=1e-12)
    phi = D.astype(np.longdouble) * (2.0 ** -39 / w.rho0)
    field = w.rho0 * 0.5 * 0.7 * float(((phi - 1.0) ** 2).sum())
    assert E[2] == pytest.approx(field, rel=1e-11)
    assert E[1] == 0.0 and E[3] == E[0] + E[2]
