"""lbm_batch_tune: the tile shapes are timed where the steps launch such tiles, and only there.  With
launches that hold all nodes, every shape times the same launch: noise chose the shape that the
checks' field snapshots and reference refreshes then ran with, after twelve times the steps."""
import pytest

pytestmark = pytest.mark.gpu

SHAPES = 12   # tile shapes


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5929_gb300 import build, lbm as L

    build.build()
    L.load()
    return L


@pytest.mark.parametrize("storage,heater,limit,nz,tuned", [
    ("f32", 0.0, False, (96, 97), False),    # k_batch_step
    ("f32", 0.3, False, (96, 97), True),     # k_batch_bulk
    ("f16", 0.0, False, (96, 97), False),    # k_batch_step16
    ("bf16", 0.0, True, (96, 128), False),   # staged tiles alone
    ("bf16", 0.0, True, (96, 97), True),     # and k_batch_bulk for odd nz
])
def test_tunes_where_tiles_are_launched(lbm, storage, heater, limit, nz, tuned):
    b = lbm.Batch([lbm.lbm_params_default(nr=40, nz=n, storage=storage, heater_len=heater) for n in nz])
    if limit:
        lbm.lbm_batch_set_wait_limit(b.b, 1 << 22)
    cols, rows, ms = b.tune(4)
    assert b.info(0).steps == (SHAPES if tuned else 1) * (2 + 4) and ms > 0
    if not tuned:
        assert (cols, rows) == (128, 1)      # the shape a batch starts with
    b.close()
