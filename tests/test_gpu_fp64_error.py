"""Round-off of one FP64 step: the one-warp-per-cell kernel, which sums and
factors differently, errs no more than the one-thread kernel, both against the
step in extended precision."""
import numpy as np
import pytest

import inputs
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


def _g(lat, order, ux, uy, th):
    """Eq. (4) for fields of shape [rows, columns]."""
    r, e = LD(lat.r), lat.e.astype(int)
    c = r * e.astype(LD)
    s = c[:, 0, None, None] * ux + c[:, 1, None, None] * uy
    u2, c2 = ux * ux + uy * uy, (c * c).sum(1)[:, None, None]
    g = 1 + s + (s * s - u2 + th * (c2 - 2)) / 2
    if order >= 4:
        g = g + s / 6 * (s * s - 3 * u2 + 3 * th * (c2 - 4))
        g = g + (s ** 4 - 6 * u2 * s * s + 3 * u2 * u2 + 6 * th * (s * s * (c2 - 6) - u2 * (c2 - 4))
                 + 3 * th * th * (c2 * c2 - 8 * c2 + 8)) / 24
    return lat.w.astype(LD)[:, None, None] * g


def _step(lat, order, thermal, Kn, u_wall, T_wall, f):
    """Eq. (5) with the Eq. (12) walls on post-collision populations f [Q][Ny][Nx]."""
    Q, Ny, Nx = f.shape
    e, r, f = lat.e.astype(int), LD(lat.r), f.astype(LD)
    m_in, gw, D = [0, 0], [], []
    for i, sg in enumerate((1, -1)):
        for b in range(Q):
            for k in range(max(0, -sg * e[b, 1])):
                m_in[i] = m_in[i] + np.roll(f[b, k if i == 0 else Ny - 1 - k], e[b, 0])
        one = np.ones((1, 1), LD)
        gw.append(_g(lat, order, one * LD(u_wall[i]), one * 0, one * (LD(T_wall[i]) - 1))[:, 0, 0])
        D.append(sum(sg * e[a, 1] * gw[i][a] for a in range(Q) if sg * e[a, 1] > 0))
    p = np.empty_like(f)
    for a in range(Q):
        for j in range(Ny):
            sj = j - e[a, 1]
            i = 0 if sj < 0 else 1
            p[a, j] = np.roll(f[a, sj] if 0 <= sj < Ny else m_in[i] * gw[i][a] / D[i], e[a, 0])
    c = r * e.astype(LD)
    rho = p.sum(0)
    ux, uy = np.tensordot(c[:, 0], p, 1) / rho, np.tensordot(c[:, 1], p, 1) / rho
    th = (np.tensordot((c * c).sum(1), p, 1) / rho - ux * ux - uy * uy) / 2 - 1 if thermal else 0 * rho
    om = 1 / (np.sqrt(2 / PI) * LD(Kn) * r * Ny / rho + LD(0.5))
    return (1 - om) * p + om * rho * _g(lat, order, ux, uy, th)


@pytest.mark.parametrize("lattice,order,thermal,Nx,Ny", [
    ("D2Q37", 4, True, 1, 500), ("D2Q25", 2, False, 8, 40), ("D2Q17", 2, False, 7, 87)])
def test_one_warp_step_errs_no_more_than_the_one_thread_step(lbm, lattice, order, thermal, Nx, Ny):
    sq = {lbm.LBM_KERNEL_CELLWARP: 0.0, lbm.LBM_KERNEL_DIRECT: 0.0}
    for seed, Kn in ((1, 0.02), (2, 0.1), (3, 0.6)):
        Tw = (1.04, 0.97) if thermal else (1.0, 1.0)
        s = lbm.Solver(lbm.Config(lattice=lattice, Nx=Nx, Ny=Ny, eq_order=order, thermal=thermal, Kn=Kn,
                                  u_wall=(-0.2, 0.25), T_wall=Tw, precision="fp64"))
        fld = [inputs.rho_field(Nx, Ny, a, seed=10 * seed + i) - b
               for i, (a, b) in enumerate(((0.05, 0.0), (0.1, 1.0), (0.05, 1.0), (0.02, 0.0)))]
        s.init_fields(fld[0], fld[1], fld[2], fld[3] if thermal else None)
        s.step(20)
        f0 = s.get_f()
        want = _step(s.lat, order, thermal, Kn, (-0.2, 0.25), Tw, f0)
        for kernel in sq:
            s.set_kernel(kernel)
            s.set_f(f0)
            s.step(1)
            sq[kernel] += float(np.mean(((s.get_f() - want) / want) ** 2))
        s.close()
    # like numbers of roundings: 5 % for chance (each a mean over 1.5e4 values and more)
    assert sq[lbm.LBM_KERNEL_CELLWARP] <= 1.05 ** 2 * sq[lbm.LBM_KERNEL_DIRECT], sq
