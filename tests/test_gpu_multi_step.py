"""GPU tests of the launches that hold their boundary nodes, and of those that take several steps
(FP32 storage): lbm_step(n) takes up to ten
steps per launch on small grids (tiles with a halo) and pairs of steps on larger ones (strips of
60 columns and chunks of rows), boundary nodes included; lbm_step(1) takes single ones.  The same
problem advanced both ways, at the sizes where that can go wrong: grids smaller than a tile, a
strip or a chunk, strip ends on, before and behind the end column for even and odd nz, chunk and
tile ends next to the walls and the axis row, and grids large enough for the marches without
boundary nodes.  The small grids also run against in-place storage, which always takes single
steps in kernels of its own.

Bounds.  FP32 storage: both ways evaluate the same formulas, rounded in another order (packed
arithmetic against scalar); the oracle parity tests' 1e-5 with their floor for fields that
vanish."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(3, 3), (3, 4), (4, 61), (5, 62), (23, 120), (23, 121), (37, 122), (41, 181), (130, 1000), (300, 701), (700, 1302)]


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5929_gb300 import build, lbm as L

    build.build()
    L.load()
    return L


def _solver(lbm, geometry, nr, nz, storage, inplace=0):
    kw = {0: dict(Ra=1e5, Da=1e-3, Pr=0.71), 1: dict(Ra=1e4, Da=5e-3, body_accel_z=2e-6),
          2: dict(Ra=0.0, tau_nu=0.8, Da=0.05, F_eps=0.0, body_accel_z=2e-6),
          3: dict(Ra=0.0, Da=1e-2, eps_mean=1.0, F_eps=0.0, Pr=0.7, tau_nu=0.62, u_in=0.05)}[geometry]
    s = lbm.Solver(lbm.lbm_params_default(nr=nr, nz=nz, geometry=geometry, storage=storage, init_noise=0.02,
                                          inplace=inplace, **kw))
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
    c = _solver(lbm, geometry, nr, nz, "f32", inplace=1)
    for n in (3, 20):       # an odd and an even count: each ends with single steps
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert a.info().steps == b.info().steps
        c.step(n)
        for x, y, z in zip(a.moments(), b.moments(), c.moments()):
            assert _err(x, y) <= 1e-5
            assert _err(x, z) <= 1e-5
        (fa, ga), (fb, gb) = a.export_populations(), b.export_populations()
        assert _err(fa, fb) <= 1e-5 and _err(ga, gb) <= 1e-5
        (ra, ma), (rb, mb) = a.residual(), b.residual()   # needs the state one step back
        assert abs(ra - rb) <= 1e-3 * rb + 1e-6 and abs(ma - mb) <= 1e-6 * abs(mb)
    for s in (a, b, c):
        s.close()


def test_batch_passes_match_single_steps(lbm):
    """The batch's launches (the nodes of every instance in one list, even and odd nz,
    every geometry, instances smaller than a block) against single steps of the same batch, with
    an odd number of steps and with captured intervals."""
    shapes = [(0, 64, 128), (0, 37, 121), (1, 23, 120), (1, 5, 61), (2, 25, 130), (3, 41, 181), (0, 3, 3), (0, 160, 320)]

    def make():
        kw = {0: dict(Ra=1e5, Da=1e-3, Pr=0.71), 1: dict(Ra=1e4, Da=5e-3, body_accel_z=2e-6),
              2: dict(Ra=0.0, tau_nu=0.8, Da=0.05, F_eps=0.0, body_accel_z=2e-6),
              3: dict(Ra=0.0, Da=1e-2, eps_mean=1.0, F_eps=0.0, Pr=0.7, tau_nu=0.62, u_in=0.05)}
        return lbm.Batch([lbm.lbm_params_default(nr=nr, nz=nz, geometry=g, init_noise=0.02, **kw[g]) for g, nr, nz in shapes])

    a, b = make(), make()
    a.step(23)
    for _ in range(23):
        b.step(1)
    a.run(20, 10, -1.0)
    for _ in range(2):
        b.rebase()
        for _ in range(10):
            b.step(1)
    assert a.info(0).steps == b.info(0).steps
    for i in range(len(shapes)):
        for x, y in zip(a.moments(i), b.moments(i)):
            assert _err(x, y) <= 1e-5, (shapes[i], _err(x, y))
    a.close()
    b.close()


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("geometry,nr,nz", [(0, 1086, 2104), (0, 1086, 2102), (1, 1086, 2102), (2, 1086, 2104),
                                            (0, 700, 1301), (1, 60, 121), (2, 61, 97), (3, 41, 181), (0, 3, 3), (0, 4, 5)])
def test_16bit_launch_with_boundary_nodes(lbm, storage, geometry, nr, nz):
    """16-bit storage: the launch that holds its boundary nodes (even nz, odd nz with its shifted
    pairs, periodic odd nz, the smallest grids) against in-place storage in the codec's error
    against FP32, and, on grids that can take it, against the staged kernel, which setting a wait
    limit selects: the same update on the same values, a flipped 16-bit rounding apart
    (test_gpu_stage's bound)."""
    n = 60
    ref, a, b = (_solver(lbm, geometry, nr, nz, sto, inplace=k) for sto, k in (("f32", 0), (storage, 0), (storage, 1)))
    for s in (ref, a, b):
        s.step(n)
    m = [s.moments() for s in (ref, a, b)]
    u = [np.stack(x[1:3]) for x in m]
    assert _err(u[1], u[0]) <= 1.5 * _err(u[2], u[0]) + 1e-5
    assert _err(m[1][3], m[0][3]) <= 1.5 * _err(m[2][3], m[0][3]) + 1e-5
    if nr > 1000:
        c = _solver(lbm, geometry, nr, nz, storage)
        lbm.lbm_set_wait_limit(c.h, (1 << 22) + 1)
        c.step(n)
        assert lbm.lbm_wait_status(c.h) == lbm.LBM_OK
        assert max(float(np.abs(np.asarray(x, np.float64) - y).max()) for x, y in zip(c.moments(), m[1])) <= 2e-5
        c.close()
    for s in (ref, a, b):
        s.close()


@pytest.mark.parametrize("storage", ["f16", "bf16"])
def test_16bit_batch_launch_matches_staged(lbm, storage):
    """The same for the batch: one launch per step from global loads against the staged tiles that a
    wait limit selects, every geometry, odd and even nz."""
    shapes = [(0, 40, 262), (0, 37, 121), (1, 21, 520), (2, 25, 130), (3, 41, 180), (0, 3, 3)]
    kw = {0: dict(Ra=1e5, Da=1e-3, Pr=0.71), 1: dict(Ra=1e4, Da=5e-3, body_accel_z=2e-6),
          2: dict(Ra=0.0, tau_nu=0.8, Da=0.05, F_eps=0.0, body_accel_z=2e-6),
          3: dict(Ra=0.0, Da=1e-2, eps_mean=1.0, F_eps=0.0, Pr=0.7, tau_nu=0.62, u_in=0.05)}
    p = [lbm.lbm_params_default(nr=nr, nz=nz, geometry=g, storage=storage, init_noise=0.02, **kw[g]) for g, nr, nz in shapes]
    a, b = lbm.Batch(p), lbm.Batch(p)
    lbm.lbm_batch_set_wait_limit(b.b, (1 << 22) + 1)
    for x in (a, b):
        x.step(61)
        x.run(20, 10, -1.0)
    assert lbm.lbm_batch_wait_status(b.b) == lbm.LBM_OK
    for i in range(len(shapes)):
        assert max(float(np.abs(np.asarray(x, np.float64) - y).max()) for x, y in zip(a.moments(i), b.moments(i))) <= 2e-5
    a.close()
    b.close()
