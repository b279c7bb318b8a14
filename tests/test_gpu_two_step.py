"""GPU tests of the two-step pass: lbm_step(n) takes pairs of steps in one launch (strips of
60 columns and chunks of rows, boundary nodes included), lbm_step(1) takes single ones.  The
same problem advanced both ways, at the sizes where the pass can go wrong: grids smaller than a
strip or a chunk, strip ends on, before and behind the end column for even and odd nz, chunk
ends next to the walls and the axis row, and grids large enough for the marches without
boundary nodes.

Bounds.  FP32 storage: both ways evaluate the same formulas, rounded in another order (packed
arithmetic against scalar); the oracle parity tests' 1e-5 with their floor for fields that
vanish.  16-bit storage: a rounding difference flips single storage roundings, so each way
carries the codec's error against FP32 storage, the pass no more than half as much again as
the single steps (the in-place tests' rule)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(3, 3), (3, 4), (4, 61), (5, 62), (23, 120), (23, 121), (37, 122), (41, 181), (130, 1000), (700, 1302)]


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5929_gb300 import build, lbm as L

    build.build()
    L.load()
    return L


def _solver(lbm, geometry, nr, nz, storage):
    kw = {0: dict(Ra=1e5, Da=1e-3, Pr=0.71), 1: dict(Ra=1e4, Da=5e-3, body_accel_z=2e-6),
          2: dict(Ra=0.0, tau_nu=0.8, Da=0.05, F_eps=0.0, body_accel_z=2e-6),
          3: dict(Ra=0.0, Da=1e-2, eps_mean=1.0, F_eps=0.0, Pr=0.7, tau_nu=0.62, u_in=0.05)}[geometry]
    s = lbm.Solver(lbm.lbm_params_default(nr=nr, nz=nz, geometry=geometry, storage=storage, init_noise=0.02, **kw))
    if geometry < 2:
        s.set_porosity(np.random.default_rng(nr * nz).uniform(0.4, 0.8, (nr, nz)).astype(np.float32))
        s.init_fields()
    return s


def _err(x, y, floor=1e-9):
    x, y = np.asarray(x, np.float64), np.asarray(y, np.float64)
    assert np.isfinite(x).all()
    return np.linalg.norm(x - y) / (np.linalg.norm(y) + floor * np.sqrt(y.size) / 1e-5)


@pytest.mark.parametrize("geometry", [0, 1, 2, 3])
@pytest.mark.parametrize("nr,nz", SHAPES)
def test_two_step_pass_matches_single_steps(lbm, geometry, nr, nz):
    a, b = _solver(lbm, geometry, nr, nz, "f32"), _solver(lbm, geometry, nr, nz, "f32")
    for n in (3, 20):       # an odd and an even count: each ends with single steps
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert a.info().steps == b.info().steps
        for x, y in zip(a.moments(), b.moments()):
            assert _err(x, y) <= 1e-5
        (fa, ga), (fb, gb) = a.export_populations(), b.export_populations()
        assert _err(fa, fb) <= 1e-5 and _err(ga, gb) <= 1e-5
        (ra, ma), (rb, mb) = a.residual(), b.residual()   # needs the state one step back
        assert abs(ra - rb) <= 1e-3 * rb + 1e-6 and abs(ma - mb) <= 1e-6 * abs(mb)
    a.close()
    b.close()


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("geometry,nr,nz", [(0, 37, 122), (0, 41, 181), (1, 23, 121), (2, 23, 120), (3, 41, 181),
                                            (0, 700, 1302), (0, 400, 1301)])
def test_two_step_pass_16bit(lbm, storage, geometry, nr, nz):
    """Across a reference refresh (after 1024 steps), which a pass must not span."""
    n = 1031
    ref, a, b = (_solver(lbm, geometry, nr, nz, sto) for sto in ("f32", storage, storage))
    ref.step(n)
    a.step(n)
    for _ in range(n):
        b.step(1)
    u = [np.stack(s.moments()[1:3]) for s in (ref, a, b)]
    T = [s.moments()[3] for s in (ref, a, b)]
    assert _err(u[1], u[0]) <= 1.5 * _err(u[2], u[0]) + 1e-5
    assert _err(T[1], T[0]) <= 1.5 * _err(T[2], T[0]) + 1e-5
    for s in (ref, a, b):
        s.close()
