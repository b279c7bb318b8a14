"""GPU tests of the two-step passes (FP32 storage, grids above a million nodes) against the FP64
oracle, in every geometry: strips of 60 columns that end on, one, two and three past a multiple of
60, even and odd nz (the lone end column), periodic columns that wrap, the pipe's axis row, inlet and
outlet, grids of a few rows, of a few columns and of one or two strips; and the benchmark's grid at
sampled nodes.  Each test counts launches, so that it fails if another kernel takes over its grids.
The batch's one-launch steps are compared with in-place storage, which runs kernels of its own.

Bounds.  FP32 arithmetic on FP32 storage: relative L2 1e-5 on rho, u and T (the parity tests' bar);
at any single node 1e-4 of the field's largest value (a few steps of FP32 rounding are some 1e-6 of
it, a wrong boundary treatment or a wrong column is 1e-2 or more)."""
import numpy as np
import pytest

from paper_1409_5929_gb300 import inputs

pytestmark = pytest.mark.gpu

GEOMETRIES = {0: dict(Ra=1e5, Da=1e-3, Pr=0.71, tau_nu=0.6), 1: dict(Ra=1e4, Da=5e-3, body_accel_z=2e-6, tau_nu=0.7),
              2: dict(Ra=0.0, tau_nu=0.8, Da=0.05, F_eps=0.0, body_accel_z=2e-6),
              3: dict(Ra=0.0, Da=1e-2, eps_mean=1.0, F_eps=0.0, Pr=0.7, tau_nu=0.62, u_in=0.05)}
# on grids of a few rows the buoyancy g beta = Ra nu alpha / L^3 and the drag nu / (Da L^2) of those
# parameters leave the model's stable range: there Ra and Da are such that both are below 0.01 a step
NARROW = dict(Ra=1.0, Da=1.0)
SHAPES = [(1000, 1020), (1003, 1021), (1002, 1022), (1001, 1023), (3, 400001), (5, 300002), (65535, 16), (60001, 17),
          (17000, 61), (9000, 121)]   # (at most 65535 rows)
W9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


@pytest.fixture(scope="module")
def lbm():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5929_gb300 import build, lbm as L

    build.build()
    L.load()
    return L


def _oparams(oracle, p):
    return oracle.params(**{k: getattr(p, k) for k in (
        "nr", "nz", "geometry", "radius_ratio", "Ra", "Da", "Pr", "J", "Ma", "tau_nu", "F_eps", "eps_mean", "T_hot",
        "T_cold", "body_accel_z", "init_noise", "seed", "u_in", "heater_len", "heater_center", "collision")}, lam=p.lam)


def _launches(lbm, s, n):
    lbm.lbm_set_timing(s.h, True)
    s.step(n)
    _, bulk, _, walls = lbm.lbm_kernel_times(s.h)
    lbm.lbm_set_timing(s.h, False)
    return bulk + walls


def _close(got, want):
    got, want = [np.stack(x) for x in (got, want)]
    for name, k in (("rho", [0]), ("u", [1, 2]), ("T", [3])):
        a, b = got[k].astype(np.float64), np.asarray(want[k], np.float64)
        assert np.isfinite(a).all()
        d = a - b
        assert np.linalg.norm(d) <= 1e-5 * np.linalg.norm(b), name
        assert np.abs(d).max() <= 1e-4 * np.abs(b).max(), (name, np.unravel_index(np.abs(d).argmax(), d.shape))


@pytest.mark.parametrize("geometry", sorted(GEOMETRIES))
@pytest.mark.parametrize("nr,nz", SHAPES)
def test_two_step_passes_match_oracle(lbm, oracle, geometry, nr, nz):
    p = lbm.lbm_params_default(nr=nr, nz=nz, geometry=geometry,
                               **{**GEOMETRIES[geometry], **(NARROW if geometry < 2 and nr < 10 else {})})
    rng = np.random.default_rng(nr + nz)
    phi = np.full((nr, nz), p.eps_mean, np.float32)
    if geometry < 2:
        phi = rng.uniform(0.4, 0.8, (nr, nz)).astype(np.float32)
    ur, uz = (rng.uniform(-0.02, 0.02, (nr, nz)).astype(np.float32) for _ in range(2))
    T = rng.uniform(0.2, 0.8, (nr, nz)).astype(np.float32)
    s = lbm.Solver(p)
    s.set_porosity(phi)
    s.init_fields(ur, uz, T)
    o = oracle.State(_oparams(oracle, p), phi=phi.astype(np.float64), ur=ur.astype(np.float64), uz=uz.astype(np.float64),
                     T=T.astype(np.float64))
    assert _launches(lbm, s, 5) == 3    # two pairs and the single step that keeps the previous state
    o.run(5)
    _close(s.moments(), o.moments())
    assert _launches(lbm, s, 4) == 3    # an even count: one pair and two single steps
    o.run(4)
    _close(s.moments(), o.moments())
    s.close()


def test_full_size_pair_at_sampled_nodes(lbm, oracle):
    """The benchmark's grid: a pair and a single step from the GPU's own state, which the oracle
    recomputes at the nodes that the sampled ones depend on."""
    nr, nz = 4096, 8192
    phi = inputs.porosity_field(nr, nz, 0.3, 0.9, 16.0, seed=2)
    p = lbm.lbm_params_default(nr=nr, nz=nz, Ra=1e6, Da=1e-4, Pr=0.71, eps_mean=float(phi.mean(dtype=np.float64)))
    s = lbm.Solver(p)
    s.set_porosity(phi)
    s.init_fields()
    s.step(20)
    rng = np.random.default_rng(1)
    samples = [(0, 0), (0, nz - 1), (nr - 1, 0), (nr - 1, nz - 1), (0, 4000), (nr - 1, 77), (1, 0), (2000, nz - 1),
               (1, 1), (nr - 2, nz - 2), (33, 59), (34, 60), (65, 8159), (66, 8160)]
    samples += [(int(a), int(b)) for a, b in zip(rng.integers(0, nr, 6), rng.integers(0, nz, 6))]
    op, r0 = _oparams(oracle, p), s.info().r0
    PHI = np.zeros((nr, nz))
    state = [(np.zeros((9, nr, nz)), np.zeros((5, nr, nz))) for _ in range(3)]   # pages are touched where used
    near = lambda x, n, h: range(max(0, x - h), min(n, x + h + 1))
    for kr in sorted({k for r, _ in samples for k in near(r, nr, 6)}):
        f, g = s.export_populations(kr, 1)
        state[0][0][:, kr], state[0][1][:, kr] = f[:, 0], g[:, 0]
        PHI[kr] = phi[kr].astype(np.float64)
    assert _launches(lbm, s, 3) == 2
    for kr, kz in samples:
        for k, h in ((1, 4), (2, 2), (3, 0)):   # a node depends on its neighbours, a boundary node on its neighbour's
            F, G = state[k - 1]
            for r in near(kr, nr, h):
                for z in near(kz, nz, h):
                    fo, go, _ = oracle.node_update(op, PHI, F, G, r, z)
                    if k < 3:
                        state[k][0][:, r, z], state[k][1][:, r, z] = fo, go
        f, g = s.export_populations(kr, 1)
        dev_o, dev_g = (x - (r0 + kr) * W9 for x in (fo, f[:, 0, kz]))
        assert np.abs(dev_g - dev_o).max() < 1e-5 * np.abs(dev_o).max()
        assert np.abs(g[:, 0, kz] - go).max() < 1e-6
    s.close()


def test_batch_steps_match_in_place_storage(lbm):
    shapes = [(0, 64, 128), (0, 37, 121), (1, 23, 120), (1, 5, 61), (2, 25, 130), (2, 3, 5), (3, 41, 181), (0, 3, 3),
              (0, 160, 320)]
    p = [lbm.lbm_params_default(nr=nr, nz=nz, geometry=g, init_noise=0.02, **GEOMETRIES[g]) for g, nr, nz in shapes]
    b = lbm.Batch(p)
    rng = np.random.default_rng(3)
    singles = []
    for i, q in enumerate(p):
        ur, uz = (rng.uniform(-0.02, 0.02, (q.nr, q.nz)).astype(np.float32) for _ in range(2))
        T = rng.uniform(0.2, 0.8, (q.nr, q.nz)).astype(np.float32)
        b.init_fields(i, ur, uz, T)
        q.inplace = 1
        s = lbm.Solver(q)
        s.init_fields(ur, uz, T)
        singles.append(s)
    b.step(23)
    for i, s in enumerate(singles):
        s.step(23)
        got, want = (np.stack(x).astype(np.float64) for x in (b.moments(i), s.moments()))
        for k in ([0], [1, 2], [3]):   # with the floor of test_gpu_multi_step.py: 1e-9 per node for fields that vanish
            n = want[k].size
            assert np.linalg.norm(got[k] - want[k]) <= 1e-5 * np.linalg.norm(want[k]) + 1e-9 * np.sqrt(n), (shapes[i], k)
        s.close()
    b.close()
