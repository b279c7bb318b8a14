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


def _kw(**kw):
    if kw["geometry"] == 2:
        kw.update(Ra=0.0, tau_nu=0.8, Da=0.05, F_eps=0.0, eps_mean=1.0, body_accel_z=1e-5)
    else:
        kw.update(Ra=1e5, Da=1e-3, Pr=0.71)
    return kw


def _compare(a_fields, b_fields):
    """The same update on the same loaded values; a multiply-add fused differently flips a 16-bit
    rounding (2^-11 of a stored deviation), nothing larger: the bound of test_gpu_stage.py."""
    for a, c in zip(a_fields, b_fields):
        a, c = np.asarray(a, np.float64), np.asarray(c, np.float64)
        assert np.isfinite(a).all() and np.isfinite(c).all()
        assert float(np.abs(a - c).max()) <= 2e-5


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("geometry", [0, 1, 2])
@pytest.mark.parametrize("nz", [2104, 2102])
def test_staged_kernel_matches_global_loads(lbm, storage, geometry, nz):
    """nz a multiple of 8 (aligned form) and 6 mod 8, ragged row and column blocks, every geometry
    class the staged kernel knows; the staged side has a limit, the other staging switched off."""
    nr = _rows(nz)
    p = lbm.lbm_params_default(**_kw(nr=nr, nz=nz, geometry=geometry, storage=storage))
    phi = np.random.default_rng(nz).uniform(0.4, 0.8, (nr, nz)).astype(np.float32) if geometry != 2 else None
    s, g = lbm.Solver(p), lbm.Solver(p)
    lbm.lbm_set_wait_limit(s.h, DEFAULT_ROUNDS)
    lbm.lbm_set_staging(g.h, False)
    for x in (s, g):
        if phi is not None:
            x.set_porosity(phi)
        x.init_fields()
    assert _staged(lbm, s, 200) and not _staged(lbm, g, 200)
    _compare(s.moments(), g.moments())
    assert lbm.lbm_wait_status(s.h) == lbm.LBM_OK
    s.close()
    g.close()


def test_staged_kernel_recovers(lbm):
    """After a wait ran out and the fields were set again, the staged kernel itself (a limit is still
    set) steps like a fresh solver's, whose limit never ran out."""
    nz = 1032
    p = lbm.lbm_params_default(nr=_rows(nz), nz=nz, Ra=1e5, Da=1e-3, Pr=0.71, storage="f16")
    s, ref = lbm.Solver(p), lbm.Solver(p)
    lbm.lbm_set_wait_limit(s.h, 0)
    s.step(1)
    assert lbm.lbm_wait_status(s.h, True) == lbm.LBM_ERR_TIMEOUT
    for x in (s, ref):
        lbm.lbm_set_wait_limit(x.h, DEFAULT_ROUNDS)
        x.init_fields()
        assert _staged(lbm, x, 50)
        assert lbm.lbm_wait_status(x.h) == lbm.LBM_OK
    _compare(s.moments(), ref.moments())
    s.close()
    ref.close()


def test_batch_staged_kernel_recovers_and_matches_global_loads(lbm):
    """The batch's staged tiles: a limit of zero runs out, so they are what runs once one is set; with
    a workable limit they step like the global-load launch of a batch that has none, graph replays
    included."""
    specs = [dict(nr=40, nz=262, geometry=0), dict(nr=37, nz=390, geometry=0, radius_ratio=3.0),
             dict(nr=21, nz=520, geometry=1, body_accel_z=2e-6), dict(nr=25, nz=646, geometry=2),
             dict(nr=30, nz=131, geometry=0), dict(nr=48, nz=96, geometry=0)]
    params = [lbm.lbm_params_default(storage="f16", **_kw(**sp)) for sp in specs]
    b, ref = lbm.Batch(params), lbm.Batch(params)
    lbm.lbm_batch_set_wait_limit(b.b, 0)
    b.step(1)
    assert lbm.lbm_batch_wait_status(b.b, True) == lbm.LBM_ERR_TIMEOUT
    ref.step(1)
    lbm.lbm_batch_set_wait_limit(b.b, DEFAULT_ROUNDS)
    for x in (b, ref):
        for i in range(len(params)):
            x.init_fields(i)
        x.step(150)
        x.run(150, 150, -1.0)
    assert lbm.lbm_batch_wait_status(b.b) == lbm.LBM_OK
    for i in range(len(params)):
        _compare(b.moments(i), ref.moments(i))
    b.close()
    ref.close()
