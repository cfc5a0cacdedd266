"""The re-emission of Eq. (12) as the FP32 step forms it (float pairs, FP64 where
their error bound does not settle the rounding) against its FP64 expression.

With a relaxation time of 1e30 steps the collision leaves a pulled population
as it is (omega f and omega g vanish in FP32), so one step stores the fills
themselves: f - w must be M_in g^w_a / D_w - w_a rounded to FP32, i.e. within
half a unit in the last place (and the FP64 expression's own round-off)."""
import numpy as np
import pytest

import inputs
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


def _expected(f, e, w, r, u_wall, Nx, Ny):
    """{(a, j): M_in(x - e_x) g^w_a / D_w} of every velocity and row filled by a wall."""
    out = {}
    for wall, u in enumerate(u_wall):
        sgn = 1 if wall == 0 else -1
        s = r * e[:, 0] * u
        g = w * (1 + s + 0.5 * (s * s - u * u))
        D = sum(sgn * e[a, 1] * g[a] for a in range(len(w)) if sgn * e[a, 1] > 0)
        m = np.zeros(Nx, dtype=np.longdouble)
        for b in range(len(w)):
            for kk in range(max(0, -sgn * e[b, 1])):
                m += np.roll(f[b, kk if wall == 0 else Ny - 1 - kk].astype(np.longdouble), e[b, 0])
        for a in range(len(w)):
            for j in range(max(0, sgn * e[a, 1])):
                out[a, j if wall == 0 else Ny - 1 - j] = np.roll(m, e[a, 0]) * (g[a] / D)
    return out


# widths below the ghost columns, at the edges of a 128-column block and of the
# x-tiles; blocks of one and of two rows; the staged kernel
@pytest.mark.parametrize("lattice", ["D2Q17", "D2Q25", "D2Q37"])
@pytest.mark.parametrize("Nx", [1, 5, 15, 17, 127, 129, 262, 700])
@pytest.mark.parametrize("kernel,variant", [(1, 0), (1, 6), (2, 0)])
def test_fp32_fills_are_the_rounded_fp64_expression(lbm, lattice, Nx, kernel, variant):
    Ny, u_wall = 7, (-0.2, 0.3)
    s = lbm.Solver(lbm.Config(lattice=lattice, Nx=Nx, Ny=Ny, eq_order=2, thermal=False, tau=1e30,
                              u_wall=u_wall, precision="fp32"))
    s.set_kernel(kernel, variant)
    s.init_fields(inputs.rho_field(Nx, Ny, 1e-2, seed=3), inputs.rho_field(Nx, Ny, 0.5, seed=4) - 1.0)
    w32 = s.lat.w.astype(np.float32).astype(np.float64)
    before = s.get_f()
    s.step(1)
    after = s.get_f()
    # g^w and D_w from the lattice's FP64 weights; storage deviates from the FP32 ones
    for (a, j), v in _expected(before, s.lat.e, s.lat.w, s.lat.r, u_wall, Nx, Ny).items():
        want = v - w32[a]
        got = after[a, j] - w32[a]
        ulp = np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
        assert np.all(np.abs(got - want) <= 0.5 * ulp + 4e-16), (a, j)
    s.close()
