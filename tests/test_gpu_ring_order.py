"""Columns of 257 to 512 rows on one CTA (one shared-memory ring per velocity)
against the same columns split over a cluster, whose CTAs hold two buffers: the
same cell updates, so the same bits, over enough chunks that a wall sum reading
a slot already stored to would show.  The step count is above what a split is
worth from, and the mean occupancy tells that one run was split and the other
was not."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu
STEPS = 130_000          # 2.5e5 row-steps per thread on one CTA: split from 125 000 on


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


def _run(lbm, reqs, cluster_rows, max_slots=16):
    s = lbm.Server(mem_budget_bytes=1 << 28, max_slots=max_slots, chunk_steps=100, cluster_rows=cluster_rows)
    ids = [s.submit(r) for r in reqs]
    s.drain(120)
    ctas = s.stats().mean_occupancy * max_slots
    res = {r.id: r for r in s.poll(len(reqs))}
    out = [(res[i].steps, res[i].residual, s.fetch(i, q.Ny)) for i, q in zip(ids, reqs)]
    s.close()
    return ctas, out


def _same(x, y):
    assert x[0] == y[0] and x[1] == y[1]
    for a, b in zip(x[2], y[2]):
        assert np.all(np.isfinite(a)) and np.array_equal(a, b)


def _req(lbm, lattice, Ny, rounding, accom=(1.0, 1.0), Kn=0.002, U=0.1):
    return lbm.make_request(lattice, Ny, Kn, U, 1.03 if lattice == "D2Q37" else 1.0, tol=1e-30,
                            max_steps=STEPS, rounding=rounding, accom=accom)


@pytest.mark.parametrize("lattice", ["D2Q17", "D2Q25", "D2Q37"])
@pytest.mark.parametrize("Ny,accom", [(257, (1.0, 1.0)), (300, (1.0, 1.0)), (509, (0.4, 1.0)),
                                      (510, (1.0, 1.0)), (511, (1.0, 1.0)), (512, (1.0, 1.0))])
@pytest.mark.parametrize("rounding", [1, 2])
def test_one_cta_is_the_split_column(lbm, lattice, Ny, accom, rounding):
    req = _req(lbm, lattice, Ny, rounding, accom)
    one, whole = _run(lbm, [req], 8192)
    split_ctas, split = _run(lbm, [req], 256)
    assert abs(one - 1.0) < 1e-9 and split_ctas > 1.9
    _same(whole[0], split[0])


def test_full_gpu_of_512_row_columns(lbm):
    import torch
    n = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    kinds = [_req(lbm, "D2Q37", 512, 0, Kn=0.002 * (1 + i), U=0.05 * (1 + i)) for i in range(4)]
    _, out = _run(lbm, [kinds[i % 4] for i in range(n)], 8192, max_slots=n)
    for i in range(4):
        _, split = _run(lbm, [kinds[i]], 256)
        for o in out[i::4]:
            _same(o, split[0])
