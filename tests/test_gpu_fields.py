"""GPU parity of the set-up and read-out kernels: f_eq from given fields
(Eq. 4), moments (Eq. 9) and mass of given populations, per lattice and
storage, on ragged grids, and the collision with and without a body force on
the same grid (the runs without one leave the source's zero terms out)."""
import numpy as np
import pytest

import workloads as W
from oracle import lbm as olbm
from oracle.lattice import get as get_lattice
from tests.parity import gpu_to_oracle_order, oracle_from_workload, rel_err

pytestmark = pytest.mark.gpu

SHAPES = [(19, (9, 11, 33)), (19, (8, 10, 130)), (9, (1, 13, 67))]
# relative size of one rounding of a stored deviation (FP64 runs are held to
# the oracle at 1e-14 in test_gpu_lbm.py)
UNIT = {"fp32": 2.0 ** -24, "fp16dev": 2.0 ** -11, "bf16dev": 2.0 ** -8}


def _ctx(ibl, q, shape, prec, force=(0.0, 0.0, 0.0)):
    grid = W.grid(shape[2], shape[1], shape[0], [W.PERIODIC] * 6, body_force=force, precision=prec)
    return ibl.from_workload({"lattice": q, "tau": 0.7, "grid": grid, "bodies": []}, init=False)


@pytest.mark.parametrize("q,shape", SHAPES)
@pytest.mark.parametrize("prec", list(UNIT))
@pytest.mark.parametrize("given", ["rest", "u", "rho_u"])
def test_init_and_readout(ibl, q, shape, prec, given):
    lat = get_lattice(q)
    rng = np.random.default_rng(3)
    u = np.zeros((lat.d,) + shape) if given == "rest" else rng.uniform(-0.05, 0.05, size=(lat.d,) + shape)
    rho = 1 + 0.02 * rng.uniform(-1, 1, size=shape) if given == "rho_u" else np.ones(shape)
    ctx = _ctx(ibl, q, shape, prec)
    ctx.ibl_init_fluid(rho if given == "rho_u" else None, None if given == "rest" else u)
    perm = gpu_to_oracle_order(ibl, q)
    f = ctx.ibl_get_populations()[perm]
    want = olbm.equilibrium(lat, rho, u)
    dev = np.abs(want - lat.w[:, None, None, None])
    # each deviation is rounded to the storage once (FP16 through FP32, below
    # 2^-24 / 2^8 in steps)
    bound = 1.01 * UNIT[prec] * dev + (2.0 ** -32 if prec == "fp16dev" else 0.0) + 4e-17
    assert (np.abs(f - want) <= bound).all()
    # read-out against the stored populations themselves
    got_rho, got_u = ctx.ibl_get_field(ibl.IBL_FIELD_RHO), ctx.ibl_get_field(ibl.IBL_FIELD_U)
    r, m = olbm.density(f), olbm.momentum(lat, f)
    assert np.abs(got_rho - r).max() < 1e-14
    assert np.abs(got_u - m / r).max() < 1e-14
    mass = ctx.ibl_mass()
    assert abs(mass - r.sum()) < 1e-13 * r.sum()
    assert mass == ctx.ibl_mass_noalloc(1024)


def test_readout_of_infinite_populations(ibl):
    q, shape = 19, (8, 8, 8)
    lat = get_lattice(q)
    f = np.tile(lat.w[:, None, None, None], (1,) + shape)
    f[0, 3, 4, 5] = np.inf
    ctx = _ctx(ibl, q, shape, "fp32")
    ctx.ibl_set_populations(f)
    rho = ctx.ibl_get_field(ibl.IBL_FIELD_RHO)
    assert np.isposinf(rho[3, 4, 5]) and np.isfinite(np.delete(rho.ravel(), (3 * 8 + 4) * 8 + 5)).all()
    assert np.isposinf(ctx.ibl_mass())


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16dev"])
@pytest.mark.parametrize("force", [(0.0, 0.0, 0.0), (0.0, 1e-5, 0.0)])
def test_collision_with_and_without_force(ibl, prec, force):
    q, shape = 19, (9, 10, 34)
    grid = W.grid(shape[2], shape[1], shape[0], [W.PERIODIC] * 6, body_force=force, precision=prec)
    cfg = {"lattice": q, "tau": 0.7, "grid": grid, "bodies": []}
    rng = np.random.default_rng(8)
    u = rng.uniform(-0.03, 0.03, size=(3,) + shape)
    ctx, sim = ibl.from_workload(cfg, init=False), oracle_from_workload(cfg)
    ctx.ibl_init_fluid(None, u)
    sim.init_fluid(u=u)
    ctx.ibl_step(5)
    sim.step(5)
    # five steps: the storage's rounding of deviations up to 0.03, a few times per step
    tol = {"fp64": 1e-13, "fp32": 5e-6, "fp16dev": 2e-2}[prec]
    assert rel_err(ctx.ibl_get_field(ibl.IBL_FIELD_U), sim.fields()[1]) < tol


# 19 FP64 populations: just under 16 MB (one copy), just over (two threads), a
# ragged last chunk, all eight threads
@pytest.mark.parametrize("shape", [(48, 48, 47), (48, 48, 49), (61, 53, 67), (79, 81, 83)])
def test_large_host_transfers_round_trip(ibl, shape):
    """Exact round trip, four contexts' transfers at once from as many threads."""
    from concurrent.futures import ThreadPoolExecutor
    lat = get_lattice(19)
    rng = np.random.default_rng(6)
    f = lat.w[:, None, None, None] * (1 + 2.0 ** -20 * rng.integers(-9999, 9999, size=(19,) + shape))
    g = np.float64(f - lat.w[:, None, None, None]) + lat.w[:, None, None, None]   # what FP64 storage holds

    def trip(k):
        ctx = _ctx(ibl, 19, shape, "fp64")
        ctx.ibl_set_populations(np.roll(f, k, axis=1))
        out = ctx.ibl_get_populations()
        return np.array_equal(out[gpu_to_oracle_order(ibl, 19)], np.roll(g, k, axis=1)[gpu_to_oracle_order(ibl, 19)])

    with ThreadPoolExecutor(4) as ex:
        assert all(ex.map(trip, range(4)))


def test_force_history_ring(ibl):
    """The asked number of most recent steps, fewer than, as many as and more than there are."""
    cfg = W.cylinder_channel(nx=64, ny=40, diameter=10.0, center=(20.0, 20.0), m=31)
    ctx = ibl.from_workload(cfg)
    ctx.ibl_step(9)
    whole = ctx.ibl_force_history(0, 9)
    assert len(whole) == 9 and np.array_equal(ctx.ibl_force_history(0, 100), whole)
    assert np.array_equal(ctx.ibl_force_history(0, 4), whole[5:]) and len(ctx.ibl_force_history(0, 0)) == 0


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_velocity_of_infinite_populations(ibl, prec):
    """u = sum c_i f_i / rho with an infinite f_0 is no number in any component (0 * inf)."""
    q, shape = 19, (8, 8, 8)
    f = np.tile(get_lattice(q).w[:, None, None, None], (1,) + shape)
    f[0, 3, 4, 5] = np.inf
    ctx = _ctx(ibl, q, shape, prec)
    ctx.ibl_set_populations(f)
    u = ctx.ibl_get_field(ibl.IBL_FIELD_U)
    assert np.isnan(u[:, 3, 4, 5]).all() and np.count_nonzero(np.isnan(u)) == 3


@pytest.mark.parametrize("prec", list(UNIT))
@pytest.mark.parametrize("q,shape", SHAPES)
def test_readout_to_fp64_accuracy(ibl, q, shape, prec):
    """rho and u of given populations as FP64 forms them: 1 + drho and the division round once each (2^-53
    relative), the sums are exact.  The deviations are multiples of 2^-13 (FP32: 2^-30) that every storage holds."""
    lat = get_lattice(q)
    rng = np.random.default_rng(12)
    top, unit = (2 ** 22, 2.0 ** -30) if prec == "fp32" else (127, 2.0 ** -14)
    k = rng.integers(-top, top + 1, size=(q,) + shape)
    ctx = _ctx(ibl, q, shape, prec)
    f = np.empty((q,) + shape)
    f[gpu_to_oracle_order(ibl, q)] = lat.w[:, None, None, None] + unit * k
    ctx.ibl_set_populations(f)
    rho, u = ctx.ibl_get_field(ibl.IBL_FIELD_RHO), ctx.ibl_get_field(ibl.IBL_FIELD_U)
    want_rho = np.longdouble(1) + k.sum(axis=0).astype(np.longdouble) * np.longdouble(unit)
    m = np.tensordot(np.asarray(lat.c)[:, :lat.d].T, k, axes=1).astype(np.longdouble) * np.longdouble(unit)
    assert (np.abs(rho - want_rho) <= 2.0 ** -53 * want_rho * 1.01).all()
    assert (np.abs(u - m / want_rho) <= 2.02 * 2.0 ** -53 * np.abs(m / want_rho)).all()


@pytest.mark.parametrize("q,shape", [(19, (160, 160, 160)), (9, (1, 1500, 2001))])
def test_init_rounds_as_fp64(ibl, q, shape):
    """FP32 storage holds f_eq - w as FP64 forms it, rounded once.  With velocities of 20 bits every FP64 operation
    but the last product is exact, so the FP32 values are determined."""
    d = get_lattice(q).d
    u = np.random.default_rng(21).integers(-2 ** 19, 2 ** 19 + 1, size=(d,) + shape) * 2.0 ** -23
    ctx = _ctx(ibl, q, shape, "fp32")
    ctx.ibl_init_fluid(None, u)
    f = ctx.ibl_get_populations()
    c, w = ibl.lattice_velocities(q)
    usq = (u * u).sum(axis=0)
    for i in range(q):
        cu = sum(int(c[i][a]) * u[a] for a in range(d))
        g = w[i] * (3 * cu + 4.5 * cu * cu - 1.5 * usq)
        # f was read as g + w in FP64, which holds all of g above 2^-20
        large = np.abs(g) > 2.0 ** -20
        assert np.array_equal((f[i] - w[i]).astype(np.float32)[large], g.astype(np.float32)[large])


def test_pinned_fields_are_copied_directly(ibl):
    """A velocity field in pinned memory goes up in one copy: the same populations as from pageable memory, and
    the call's processor time stays near one thread's (staged through the pinned chunks, several threads copy)."""
    import time
    torch = pytest.importorskip("torch")
    shape = (160, 160, 160)
    pinned = torch.empty((3,) + shape, dtype=torch.float64).pin_memory().numpy()
    pinned[:] = np.random.default_rng(5).uniform(-0.05, 0.05, size=pinned.shape)
    ctx = _ctx(ibl, 19, shape, "fp32")
    ctx.ibl_init_fluid(None, pinned.copy())
    want = ctx.ibl_get_field(ibl.IBL_FIELD_U)
    ratios = []
    for _ in range(6):
        cpu, wall = time.process_time(), time.perf_counter()
        ctx.ibl_init_fluid(None, pinned)
        ratios.append((time.process_time() - cpu) / (time.perf_counter() - wall))
    assert np.array_equal(ctx.ibl_get_field(ibl.IBL_FIELD_U), want)
    assert min(ratios) < 1.5
