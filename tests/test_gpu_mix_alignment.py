"""Mode mixing of the warm-start network on arrays that start at any float: parameters sit one behind
another in one buffer, in the order the caller lists them, and a C caller may pass any float pointer.
The sums are the same in the same order whatever the width of the loads, so results are equal to the
aligned call's bit by bit."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fno():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5929_gb300 import build, fno as F

    build.build()
    F.load()
    return F


def _at(values, offset):
    """The values in device memory, `offset` floats past a 256-byte boundary."""
    import torch

    buf = torch.full((values.size + 8,), 7.0, device="cuda")
    view = buf[offset:offset + values.size].view(values.shape)
    view.copy_(torch.from_numpy(values))
    assert view.data_ptr() % 16 == 4 * offset % 16
    return view


@pytest.mark.parametrize("C,B", [(32, 1), (32, 5), (64, 8)])
@pytest.mark.parametrize("offsets", [(1, 0, 0), (0, 1, 0), (0, 2, 0), (0, 3, 0), (0, 0, 1), (2, 3, 1), (3, 1, 2)])
def test_any_float_alignment(fno, C, B, offsets):
    import torch

    M, rng = 8, np.random.default_rng(C + B)
    dims = fno.fno_net_dims(B, 64, 128, C, M, 128, 8, 3)
    lib, dp, s = fno.load_net(), ctypes.byref(dims), torch.cuda.current_stream().cuda_stream
    W, dY = (rng.normal(size=(M, 2 * M, 2, B, C)).astype(np.float32) for _ in range(2))
    R, dR0 = (rng.normal(size=(2 * M, M, C, C, 2)).astype(np.float32) for _ in range(2))

    def run(ow, orr, od):
        w, r, dy, dr = _at(W, ow), _at(R, orr), _at(dY, od), _at(dR0, orr)
        y, dw = _at(np.zeros_like(W), od), _at(np.zeros_like(W), ow)
        fno._ncheck(lib.fno_net_mix_fwd(dp, w.data_ptr(), r.data_ptr(), y.data_ptr(), s))
        fno._ncheck(lib.fno_net_mix_bwd(dp, w.data_ptr(), r.data_ptr(), dy.data_ptr(), dw.data_ptr(), dr.data_ptr(), 1, s))
        out = [y.cpu(), dw.cpu(), dr.cpu()]
        fno._ncheck(lib.fno_net_mix_bwd(dp, w.data_ptr(), r.data_ptr(), dy.data_ptr(), dw.data_ptr(), dr.data_ptr(), 0, s))
        return out + [dr.cpu()]

    for a, b in zip(run(*offsets), run(0, 0, 0)):
        assert torch.equal(a, b)


def test_parameters_in_any_order(fno):
    """q2 (three floats) listed first puts every later parameter of the flat buffer off alignment."""
    import torch

    sizes = dict(nr=64, nz=128, width=32, modes=8, layers=2, in_ch=8, out_ch=3, hidden=128)
    P = fno.init_params(seed=4, **sizes)
    Q = {"q2": P["q2"], **{k: v for k, v in P.items() if k != "q2"}}
    assert P["q2"].size % 4
    x = torch.randn((3, 64, 128, 8), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    t = torch.randn((3, 64, 128, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    a, b = (fno.FusedFNO2d(params=p, **sizes) for p in (P, Q))
    assert b.w["R0"].data_ptr() % 8
    ya, yb = a.forward(x).clone(), b.forward(x).clone()
    assert torch.equal(ya, yb)
    for net in (a, b):
        net.zero_grad()
        net.loss_and_grad(x, t)
    torch.cuda.synchronize()
    assert fno.fno_net_status(True) == 0
    for k in P:   # gradients are summed with atomics: their last bits vary from run to run
        ga, gb = a.g[k].double(), b.g[k].double()
        assert float((ga - gb).norm()) <= 1e-4 * float(ga.norm()) + 1e-12, k
