"""lbm_step under CUDA graph capture: replays of a captured even number of steps advance the problem as
the same calls do, in every kernel that serves two-buffer problems.  Launches alternate between the two
buffers, so that takes an even number of launches whatever the steps per launch; outside capture the
plan is free (and takes fewer launches)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5929_gb300 import build, lbm as L

    build.build()
    L.load()
    return L


@pytest.mark.parametrize("nr,nz,storage", [(48, 96, "f32"), (100, 200, "f32"), (300, 701, "f32"), (1003, 1021, "f32"),
                                           (100, 201, "f16")])
@pytest.mark.parametrize("n", [2, 4, 6, 8, 10, 18])
def test_replays_continue(lbm, nr, nz, storage, n):
    import torch

    p = lbm.lbm_params_default(nr=nr, nz=nz, Ra=1e5, Da=1e-3, storage=storage, init_noise=0.02)
    a, b = lbm.Solver(p), lbm.Solver(p)
    stream = torch.cuda.Stream()
    lbm.lbm_set_stream(a.h, stream.cuda_stream)
    for s in (a, b):
        s.step(3)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        a.step(n)
    with torch.cuda.stream(stream):
        for _ in range(3):
            g.replay()
    torch.cuda.synchronize()
    for _ in range(3):
        b.step(n)
    # FP32 rounding of other launch sizes; the flow itself moves by far more in n steps
    for x, y in zip(a.moments(), b.moments()):
        x, y = np.asarray(x, np.float64), np.asarray(y, np.float64)
        assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y) + 1e-9 * np.sqrt(y.size)
    a.close()
    b.close()
