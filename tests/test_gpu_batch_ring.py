"""One-CTA columns kept in one shared-memory ring per velocity (257 to 512 rows;
509 where a wall reflects specularly) against the same columns split over a
cluster, whose CTAs hold two buffers, and in L2 beyond: the same cell updates,
so the same bits."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


def _run(lbm, req, steps, cluster_rows):
    s = lbm.Server(mem_budget_bytes=1 << 28, max_slots=16, chunk_steps=50, cluster_rows=cluster_rows)
    rid = s.submit(lbm.make_request(*req, tol=1e-30, max_steps=steps[0], rounding=steps[1], accom=steps[2]))
    s.drain(120)
    r = s.poll(4)[0]
    out = s.fetch(rid, req[1])
    s.close()
    return r, out


@pytest.mark.parametrize("lattice", ["D2Q17", "D2Q25", "D2Q37"])
@pytest.mark.parametrize("Ny", [257, 509, 510, 512, 513])
@pytest.mark.parametrize("accom", [(1.0, 1.0), (0.4, 1.0)])
@pytest.mark.parametrize("rounding", [1, 2])
def test_ring_is_the_split_column(lbm, lattice, Ny, accom, rounding):
    # more steps than the ring has slots; Kn small: the request may be split
    req = (lattice, Ny, 0.002, 0.1, 1.03 if lattice == "D2Q37" else 1.0)
    steps = (700, rounding, accom)
    whole, a = _run(lbm, req, steps, 8192)
    split, b = _run(lbm, req, steps, 256)
    assert whole.steps == split.steps and whole.residual == split.residual
    for x, y in zip(a, b):
        assert np.all(np.isfinite(x)) and np.array_equal(x, y)
