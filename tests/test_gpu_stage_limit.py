"""16-bit storage: which launch a step takes.  Grids up to eight million nodes take one launch from
global loads unless a wait limit was set, whatever its value; then, and on larger grids, the staged
kernel runs, with the wall kernel beside it (so lbm_kernel_times counts wall launches)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DEFAULT_ROUNDS = 1 << 22   # STAGE_SPIN: the value that the default happens to have


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5929_gb300 import build, lbm as L

    build.build()
    L.load()
    return L


def _rows(nz):
    """Rows at which nz columns give 16 blocks of 256 columns and 4 rows per SM, and two more."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return 4 * -(-16 * sms // -(-nz // 256)) + 2


def _staged(lbm, s, n=1):
    """Whether the next n steps run the staged kernel: it is followed by the wall kernel."""
    lbm.lbm_set_timing(s.h, True)
    s.step(n)
    _, bulk, _, walls = lbm.lbm_kernel_times(s.h)
    lbm.lbm_set_timing(s.h, False)
    assert bulk == n and walls in (0, n)
    return walls == n


@pytest.mark.parametrize("rounds", [DEFAULT_ROUNDS, DEFAULT_ROUNDS - 1, 2 * DEFAULT_ROUNDS])
def test_any_limit_selects_the_staged_kernel(lbm, rounds):
    nz = 1032
    s = lbm.Solver(lbm.lbm_params_default(nr=_rows(nz), nz=nz, Ra=1e4, storage="f16"))
    assert not _staged(lbm, s)
    lbm.lbm_set_wait_limit(s.h, rounds)
    assert _staged(lbm, s, 2)
    lbm.lbm_set_staging(s.h, False)
    assert not _staged(lbm, s)
    lbm.lbm_set_staging(s.h, True)
    lbm.lbm_set_wait_limit(s.h, -1)
    assert not _staged(lbm, s)
    assert lbm.lbm_wait_status(s.h) == lbm.LBM_OK
    s.close()
