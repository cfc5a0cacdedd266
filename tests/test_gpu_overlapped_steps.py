"""Step launches that overlap (programmatic dependent launch: several steps'
blocks are resident at once on a small grid) against the same steps with the
stream waited for after each: the same bits, in plain launches and in replayed
graphs."""
import numpy as np
import pytest

import inputs
from gpu_util import need_gpu, order_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16dev", "bf16shift"])
@pytest.mark.parametrize("kernel,variant", [(1, 0), (1, 6), (3, 0)])
@pytest.mark.parametrize("lattice,Nx,Ny", [("D2Q37", 9, 16), ("D2Q17", 130, 7), ("D2Q37", 600, 33),
                                           ("D2Q25", 4300, 12)])
def test_overlapped_steps_are_the_steps_in_turn(lbm, precision, kernel, variant, lattice, Nx, Ny):
    o, t = order_for(lattice)
    a, b = (lbm.Solver(lbm.Config(lattice=lattice, Nx=Nx, Ny=Ny, eq_order=o, thermal=t, Kn=0.06,
                                  u_wall=(-0.2, 0.25), precision=precision)) for _ in range(2))
    rho = inputs.rho_field(Nx, Ny, 1e-2, seed=5)
    for s in (a, b):
        s.set_kernel(kernel, variant)
        s.init_fields(rho)
    for n in (63, 150):
        a.step(n)
        a.sync()
        for _ in range(n):
            b.step(1)
            b.sync()
        assert np.array_equal(a.get_f(), b.get_f())
    a.close(), b.close()
