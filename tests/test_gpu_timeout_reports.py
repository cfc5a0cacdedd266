"""A step kernel whose bounded wait runs out leaves an incomplete state.  Every
call that hands out that state, or what is computed from it, reports it, once;
the reloaded solver steps on like one that never failed."""
import numpy as np
import pytest

import inputs
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


READ_OUTS = {
    "sync": lambda s: s.sync(),
    "get_f": lambda s: s.get_f(),
    "get_state": lambda s: s.get_state(),
    "macros": lambda s: s.macros(),
    "fluxes": lambda s: s.fluxes(),
    "wall_mass": lambda s: s.wall_mass(),
    "stats": lambda s: s.stats(),
}


def _solvers(lbm, n, **kw):
    args = dict(lattice="D2Q17", Nx=70, Ny=12, eq_order=2, thermal=False, Kn=0.08,
                u_wall=(-0.1, 0.15), precision="fp64")
    return [lbm.Solver(lbm.Config(**{**args, **kw})) for _ in range(n)]


def _expire_and_recover(lbm, a, b, read, rho, steps):
    """a's waits give up; `read` reports it; reloaded, a is b bit for bit."""
    a.init_fields(rho)
    a.set_wait_limit(0)
    a.step(3)
    with pytest.raises(lbm.LBMError) as ei:
        read(a)
    assert ei.value.status == lbm.LBM_ETIMEOUT
    read(a)                                      # reported once
    a.set_wait_limit(2_000_000_000)
    for s in (a, b):
        s.init_fields(rho)
        for n in steps:
            s.step(n)
    assert np.array_equal(a.get_f(), b.get_f())
    a.close(), b.close()


@pytest.mark.parametrize("call", READ_OUTS)
def test_staged_timeout_is_reported_by_every_read_out(lbm, call):
    a, b = _solvers(lbm, 2)
    for s in (a, b):
        s.set_kernel(lbm.LBM_KERNEL_STAGED, 0)
    _expire_and_recover(lbm, a, b, READ_OUTS[call], inputs.rho_field(70, 12, 1e-2, seed=8), (5,))


# more than 64 cells: the whole-chip launch with a grid barrier, one block to many
@pytest.mark.parametrize("Nx,Ny", [(5, 13), (1, 500), (60, 60)])
def test_fp64_grid_barrier_wait_limit(lbm, Nx, Ny):
    a, b = _solvers(lbm, 2, Nx=Nx, Ny=Ny)
    for s in (a, b):
        s.set_kernel(lbm.LBM_KERNEL_CELLWARP)
    # several launches afterwards: the barrier's words were left as it needs them
    _expire_and_recover(lbm, a, b, READ_OUTS["macros"], inputs.rho_field(Nx, Ny, 1e-2, seed=8),
                        (7, 2, 33, 2100))
