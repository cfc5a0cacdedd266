"""The autotuner's choice against the candidates it chose from."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


def _us(s, n, best_of=5):
    import torch
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    s.step(n)
    us = []
    for _ in range(best_of):
        e0.record(s.stream)
        s.step(n)
        e1.record(s.stream)
        e1.synchronize()
        us.append(e0.elapsed_time(e1) * 1e3 / n)
    return min(us)


def _solver(lbm, **kw):
    import torch
    args = dict(lattice="D2Q37", eq_order=3, thermal=True, Kn=0.06, u_wall=(-0.2, 0.2), noise_amp=1e-3)
    return lbm.Solver(lbm.Config(**{**args, **kw}), stream=torch.cuda.Stream())


def test_fp64_tuner_times_the_many_step_launches(lbm):
    # one launch per step 19 us, many per launch 13, one thread per cell 18
    s = _solver(lbm, Nx=50, Ny=60, precision="fp64")
    s.autotune(10)
    tuned = _us(s, 400)
    s.set_kernel(lbm.LBM_KERNEL_CELLWARP)
    warp = _us(s, 400)
    s.close()
    assert tuned <= 1.15 * warp


# wide grids below the line by cells, where one warp per cell is the slower kernel
@pytest.mark.parametrize("lattice,Nx,Ny,precision", [
    ("D2Q37", 122, 41, "fp32"), ("D2Q37", 224, 22, "fp32"), ("D2Q37", 212, 21, "fp32"),
    ("D2Q25", 200, 20, "fp32"), ("D2Q17", 141, 16, "bf16shift")])
def test_wide_grids_are_not_held_on_the_slower_kernel(lbm, lattice, Nx, Ny, precision):
    o, t = (3, True) if lattice == "D2Q37" else (2, False)
    s = _solver(lbm, lattice=lattice, Nx=Nx, Ny=Ny, precision=precision, eq_order=o, thermal=t)
    s.autotune(10)
    tuned = _us(s, 400)
    s.set_kernel(lbm.LBM_KERNEL_DIRECT)
    direct = _us(s, 400)
    s.close()
    assert tuned <= 1.25 * direct


def test_a_size_class_across_the_line_keeps_both_choices(lbm):
    # 70 x 60 and 128 x 64: one class, on either side of the line
    small = _solver(lbm, Nx=70, Ny=60, precision="fp32")
    large = _solver(lbm, Nx=128, Ny=64, precision="fp32")
    first = small.autotune(10), large.autotune(10)
    assert (small.autotune(10), large.autotune(10)) == first
    small.close(), large.close()


@pytest.mark.parametrize("precision,n", [("fp64", 8), ("fp32", 9), ("bf16dev", 9), ("bf16shift", 9)])
@pytest.mark.parametrize("lattice,Nx", [("D2Q37", 300), ("D2Q37", 600), ("D2Q25", 300)])
def test_the_shape_without_a_register_request_is_a_variant(lbm, precision, n, lattice, Nx):
    # FP32 and BF16 variant 0 asks for registers by format and lattice; the
    # shape that asks for none is the last variant, the same step bit for bit
    o, t = (3, True) if lattice == "D2Q37" else (2, False)
    a, b = (_solver(lbm, lattice=lattice, Nx=Nx, Ny=20, precision=precision, eq_order=o, thermal=t)
            for _ in range(2))
    assert a.variant_count(lbm.LBM_KERNEL_DIRECT) == n
    for s, v in ((a, 0), (b, n - 1)):
        s.set_kernel(lbm.LBM_KERNEL_DIRECT, v)
        s.init()
        s.step(20)
    assert np.array_equal(a.get_f(), b.get_f())
    a.close(), b.close()
