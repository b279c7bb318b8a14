"""The reference refresh of an FP32 batch run (one launch for all instances, blocks by the largest)
against lbm_batch_rebase's (a launch per instance), on instances of one block, of a block's edge and of
many blocks beside each other: the same update of each node, to FP32 rounding (2^-24 relative per
operation; 1e-6 in L2)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [[(3, 3)], [(33, 31), (32, 32), (25, 41), (4, 4)], [(1501, 1400), (3, 5), (48, 96)]])
def test_run_refreshes_as_rebase_does(shapes):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5929_gb300 import build, lbm

    build.build()
    p = [lbm.lbm_params_default(nr=nr, nz=nz, Ra=1e4, init_noise=0.1, tau_nu=0.6) for nr, nz in shapes]
    a, b = lbm.Batch(p), lbm.Batch(p)
    for x in (a, b):
        x.step(7)
    a.run(6, 2, -1.0)
    for _ in range(3):
        b.rebase()
        b.step(2)
    for i in range(len(p)):
        for x, y in zip(a.moments(i), b.moments(i)):
            x, y = np.asarray(x, np.float64), np.asarray(y, np.float64)
            assert np.isfinite(x).all() and np.linalg.norm(x - y) <= 1e-6 * np.linalg.norm(y) + 1e-12
    a.close()
    b.close()
