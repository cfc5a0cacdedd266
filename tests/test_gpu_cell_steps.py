"""Many FP64 steps of a small grid in one launch (a cluster's shared memory up
to 64 cells, the whole chip up to 28 cells per SM, a launch per step beyond)
against the same steps one call at a time: the same arithmetic on the same
values, so the populations agree bit for bit; and the state that is left, its
halo copies included, steps on alike under the direct kernel."""
import numpy as np
import pytest

import inputs
from gpu_util import need_gpu, order_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


def _solver(lbm, lattice, Nx, Ny, **kw):
    o, t = order_for(lattice)
    args = dict(lattice=lattice, Nx=Nx, Ny=Ny, eq_order=o, thermal=t, Kn=0.07, u_wall=(-0.2, 0.25),
                T_wall=(1.04, 0.97), precision="fp64", kernel=lbm.LBM_KERNEL_CELLWARP)
    s = lbm.Solver(lbm.Config(**{**args, **kw}))
    s.init_fields(inputs.rho_field(Nx, Ny, 1e-2, seed=6))
    return s


# cells at the edges of the launch shapes: one CTA, a full cluster and one
# more cell, one warp per SM sub-partition and one more cell, the widest block
# and past it
@pytest.mark.parametrize("lattice,Nx,Ny", [("D2Q37", 1, 6), ("D2Q25", 1, 64), ("D2Q17", 5, 13),
                                           ("D2Q37", 8, 76), ("D2Q37", 7, 87), ("D2Q25", 64, 64),
                                           ("D2Q17", 64, 67)])
@pytest.mark.parametrize("n", [7, 8])
def test_one_launch_is_the_same_as_one_call_per_step(lbm, lattice, Nx, Ny, n):
    a, b = _solver(lbm, lattice, Nx, Ny), _solver(lbm, lattice, Nx, Ny)
    a.step(n)
    for _ in range(n):
        b.step(1)
    a.sync()
    assert np.array_equal(a.get_f(), b.get_f())
    for s in (a, b):
        s.set_kernel(lbm.LBM_KERNEL_DIRECT, 0)
        s.step(1)
    assert np.array_equal(a.get_f(), b.get_f())
    a.close(), b.close()


@pytest.mark.parametrize("kw", [dict(accom=(0.3, 1.0)), dict(tau=0.02), dict(mu_exp=0.7),
                                dict(eq_order=3), dict(eq_order=2), dict(thermal=False)])
@pytest.mark.parametrize("Nx,Ny", [(3, 9), (9, 31)])
def test_options(lbm, kw, Nx, Ny):
    a, b = _solver(lbm, "D2Q37", Nx, Ny, **kw), _solver(lbm, "D2Q37", Nx, Ny, **kw)
    a.step(12)
    for _ in range(12):
        b.step(1)
    assert np.array_equal(a.get_f(), b.get_f())
    # the one-thread kernel sums in another order: round-off of 12 steps
    b.set_kernel(lbm.LBM_KERNEL_DIRECT, 0)
    b.init_fields(inputs.rho_field(Nx, Ny, 1e-2, seed=6))
    b.step(12)
    fa, fb = a.get_f(), b.get_f()
    assert np.max(np.abs(fa - fb) / np.abs(fb)) < 1e-12
    a.close(), b.close()


@pytest.mark.parametrize("Nx,Ny", [(1, 40), (5, 40)])
def test_steps_in_a_captured_graph(lbm, Nx, Ny):
    import torch
    stream = torch.cuda.Stream()
    o, t = order_for("D2Q25")
    cfg = lbm.Config(lattice="D2Q25", Nx=Nx, Ny=Ny, eq_order=o, thermal=t, Kn=0.07, precision="fp64")
    rho = inputs.rho_field(Nx, Ny, 1e-2, seed=6)
    a, b = lbm.Solver(cfg, stream=stream), lbm.Solver(cfg)
    a.init_fields(rho), b.init_fields(rho)
    a.step(8)
    a.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        a.step(8)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    b.step(32)
    assert np.array_equal(a.get_f(), b.get_f())
    a.close(), b.close()
