"""The batched-path autotuner times a lone column on the clusters it reports, and
takes no chunk that outlasts a launch."""
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


def test_lone_columns_and_chunk_length(lbm):
    import torch
    cfg = lbm.lbm_server_cfg_default()
    cfg.mem_budget_bytes = 1 << 28
    cfg.max_slots = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    rep = lbm.lbm_server_autotune(cfg)
    for us in rep["lone_us"]:
        assert all(t > 0 for t in us[0][:4])
        # 1024 rows: 8 CTAs have half the rows of 4; a column that the server
        # had not split as asked would give both the same time
        assert us[1][3] < 0.95 * us[1][2], us[1]
        # 4096 rows: each doubling up to 16 CTAs shortens the step
        assert all(b < 0.95 * a for a, b in zip(us[2], us[2][1:])), us[2]
    # a chunk of the columns that the rates were taken of (256 rows of D2Q37: 333 /
    # 74 times chunk_steps) on the full GPU lasts 2 ms at most
    rate = dict(zip(rep["chunk_try"], rep["chunk_glups"]))[cfg.chunk_steps]
    assert round(cfg.chunk_steps * 333 / 74) * 256 * cfg.max_slots / rate <= 2e6
