"""The batched walls' re-emission c0 + d c in floats (csrc/float_pairs.h, built
for the host) against exact rationals: it errs by no more than the FP64
expression it stands for, over the deviations, wall speeds and temperatures of
the requests."""
import ctypes as C
import os
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

from paper_1209_5201_gb300 import lbm

CSRC = os.path.join(os.path.dirname(lbm.__file__), "csrc")
SRC = r"""
#include "float_pairs.h"
using namespace lbm;
// the terms as a group of four lanes sums them: every fourth each, then two
// exchanges; hi + lo of lane `lane`
extern "C" void emit(const float *d, int n, double c, double W, double w, int lane, float *out) {
    Sum3 s[4], t[4];
    for (int l = 0; l < 4; ++l)
        for (int i = l; i < 28; i += 4) s[l].add(i < n ? d[i] : 0.0f);
    for (int o = 1; o <= 2; o <<= 1) {
        for (int l = 0; l < 4; ++l) t[l] = s[l];
        for (int l = 0; l < 4; ++l) s[l].add(t[l ^ o].h, t[l ^ o].m, t[l ^ o].l);
    }
    emit3(emit3_of(c, W, w), s[lane], out[0], out[1]);
}
"""


@pytest.fixture(scope="module")
def emit(tmp_path_factory):
    d = tmp_path_factory.mktemp("pairs")
    (d / "pairs.cpp").write_text(SRC)
    so = str(d / "pairs.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-o", so,
                    str(d / "pairs.cpp")], check=True)
    fn = C.CDLL(so).emit
    fn.argtypes = [C.POINTER(C.c_float), C.c_int, C.c_double, C.c_double, C.c_double, C.c_int,
                   C.POINTER(C.c_float)]
    fn.restype = None
    return fn


def _shape(lat, u, th, order):
    """g^eq / w at velocity (u, 0), temperature 1 + th."""
    e, r = lat.e, lat.r
    c2, s, u2 = r * r * (e[:, 0] ** 2 + e[:, 1] ** 2), r * e[:, 0] * u, u * u
    g = 1 + s + 0.5 * (s * s - u2 + th * (c2 - 2))
    if order >= 4:
        g += s / 6 * (s * s - 3 * u2 + 3 * th * (c2 - 4))
        g += (s ** 4 - 6 * u2 * s * s + 3 * u2 * u2 + 6 * th * (s * s * (c2 - 6) - u2 * (c2 - 4))
              + 3 * th * th * (c2 * c2 - 8 * c2 + 8)) / 24
    return g


@pytest.mark.parametrize("lattice,order", [("D2Q17", 2), ("D2Q25", 2), ("D2Q37", 4)])
def test_re_emission_errs_no_more_than_fp64(emit, lattice, order):
    lat, rng = lbm.Lattice(lattice), np.random.default_rng(1)
    w, ey = lat.w.astype(np.float32), lat.e[:, 1]
    terms = [a for a in range(len(w)) for _ in range(max(0, -ey[a]))]
    out = [a for a in range(len(w)) if ey[a] > 0]
    W = float(sum(np.float64(w[a]) for a in terms))
    sq, most = [0.0, 0.0], [0.0, 0.0]
    for _ in range(400):
        th = (lambda: rng.uniform(-0.1, 0.1)) if order == 4 else (lambda: 0.0)
        g = lat.w * _shape(lat, rng.uniform(-0.3, 0.3), th(), order)
        D = sum(ey[a] * g[a] for a in out)
        f = rng.uniform(0.95, 1.05) * _shape(lat, rng.uniform(-0.3, 0.3), th(), order) - 1
        f *= 1 + 10.0 ** rng.uniform(-4, -1) * rng.normal(size=len(w))
        d = np.array([lat.w[a] * f[a] for a in terms], dtype=np.float32)
        exact_d, lanes = sum(F(float(x)) for x in d), np.zeros(32)
        lanes[:len(d)], lanes[len(d)] = d, W         # a butterfly over a warp, in FP64
        for o in (16, 8, 4, 2, 1):
            lanes = lanes + lanes[np.arange(32) ^ o]
        for a in out:
            c, hl = float(g[a] / D), (C.c_float * 2)()
            exact = (exact_d + F(W)) * F(c) - F(float(w[a]))
            x = float(F(float(lanes[0])) * F(c) - F(float(w[a])))      # one rounding: an FMA
            hi = np.float32(x)
            fp64 = F(float(hi)) + F(float(np.float32(x - float(hi))))
            emit(d.ctypes.data_as(C.POINTER(C.c_float)), len(d), c, W, float(w[a]), a % 4, hl)
            assert np.float32(hl[0] + hl[1]) == np.float32(hl[0])      # lo: the remainder of hi
            for i, v in enumerate((fp64, F(hl[0]) + F(hl[1]))):
                err = abs(float(v - exact)) / float(w[a])
                sq[i] += err * err
                most[i] = max(most[i], err)
    # the same rounding of the remainder, and sums of like size: 2 % for chance
    assert sq[1] <= 1.02 ** 2 * sq[0] and most[1] <= 1.1 * most[0], (sq, most)
