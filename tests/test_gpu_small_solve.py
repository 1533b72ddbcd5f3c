"""GPU parity of the IB step of small marker sets, whose kinematics, band and
implicit solve run on one thread-block cluster: marker counts around the
changes of the cluster's size (72 rows a block), odd counts, a third body of a
single marker (a row pair across two bodies), bodies whose stencils share band
tiles, against k_pcg on the same run (an explicit dense preconditioner) and
the oracle."""
import numpy as np
import pytest

import workloads as W
from tests.parity import TOL_FIELD_FP64, compare_fields, oracle_from_workload, rel_err

pytestmark = pytest.mark.gpu


def _wings(chord, extra, prec="fp64"):
    cfg = W.clap_fling_3d(nx=40, ny=36, nz=48, chord=chord, Re=10.0, J=0.1, period=900.0, precision=prec,
                          faces="periodic", phase=0.7)
    if extra:
        b = dict(cfg["bodies"][0])
        b.update(X0=np.zeros((1, 3)), ds=np.ones(1), origin=(30.0, 9.3, 17.6), hinge=(0.0, 0.0, 0.0))
        cfg["bodies"] = cfg["bodies"] + [b]
    return cfg


# chord -> 2 x 44, 2 x 68 + 1, 2 x 144 + 1, 2 x 248 markers: 2, 2, 8 and 8 blocks
@pytest.mark.parametrize("chord,extra", [(3.2, False), (4.0, True), (6.0, True), (7.9, False)])
def test_cluster_solve_matches_general_and_oracle(ibl, chord, extra):
    cfg = _wings(chord, extra)
    a, b = ibl.from_workload(cfg), ibl.from_workload(cfg)
    b.ibl_solver_preconditioner(0, -1)
    sim = oracle_from_workload(cfg)
    for c in (a, b):
        c.ibl_step(12)
    sim.step(12)
    compare_fields(a, sim, ibl, TOL_FIELD_FP64)
    # both solves stop at a relative residual of 1e-10
    assert rel_err(a.ibl_get_field(ibl.IBL_FIELD_U), b.ibl_get_field(ibl.IBL_FIELD_U)) < TOL_FIELD_FP64
    again = ibl.from_workload(cfg)
    again.ibl_step(12)
    assert np.array_equal(again.ibl_get_populations(), a.ibl_get_populations())


def test_one_marker_and_moving_band(ibl):
    """One marker crossing several tiles and a periodic face: the band follows it."""
    m = {"kind": W.WAVE_COS, "amp": 9.0, "offset": 0.0}
    body = {"X0": np.zeros((1, 2)), "ds": np.ones(1), "hinge": (0, 0, 0), "axis": (0, 0, 1), "origin": (30.0, 7.4, 0.0),
            "A": m, "alpha": {"kind": W.WAVE_CONST, "amp": 0.0, "offset": 0.0}, "beta": 0.3, "phi": 0.0, "f": 1 / 300.0,
            "J": 0.0}
    cfg = {"lattice": 9, "tau": 0.8, "grid": W.grid(35, 40, 1, [W.PERIODIC] * 6, precision="fp64"), "bodies": [body],
           "u0": (0.0, 0.0, 0.0), "reference": {"U_ref": 0.1, "L": 1.0, "rho_ref": 1.0}}
    ctx, sim = ibl.from_workload(cfg), oracle_from_workload(cfg)
    ctx.ibl_step(150)
    sim.step(150)
    compare_fields(ctx, sim, ibl, TOL_FIELD_FP64)
    force = ctx.ibl_get_field(ibl.IBL_FIELD_FORCE)
    assert 0 < np.count_nonzero(force[0]) <= 16   # only the last step's stencil


def test_marker_list_capacity_without_lists(ibl):
    """576 markers of one still body on one 16 x 16 tile (a list holds 512): refused at the first step, although
    nothing reads the lists of a single body."""
    g = 14.1 + 0.79 * np.arange(24)
    X0 = np.stack([a.ravel() for a in np.meshgrid(g, g)], axis=1)
    still = {"kind": W.WAVE_CONST, "amp": 0.0, "offset": 0.0}
    body = {"X0": X0, "ds": np.ones(len(X0)), "hinge": (0, 0, 0), "axis": (0, 0, 1), "origin": (0.0, 0.0, 0.0),
            "A": still, "alpha": still, "beta": 0.0, "phi": 0.0, "f": 1 / 300.0, "J": 0.0}
    cfg = {"lattice": 9, "tau": 0.8, "grid": W.grid(48, 48, 1, [W.PERIODIC] * 6, precision="fp64"), "bodies": [body],
           "u0": (0.0, 0.0, 0.0), "reference": {"U_ref": 0.1, "L": 1.0, "rho_ref": 1.0}}
    ctx = ibl.from_workload(cfg)
    with pytest.raises(ibl.IblError, match="IBL_EINVAL"):
        ctx.ibl_step(1)
        ctx.ibl_sync()
    # 528 markers at 1.5 lattice units spread over nine tiles: the same calls run
    body["X0"] = np.stack([a.ravel() for a in np.meshgrid(6.0 + 1.5 * np.arange(22), 6.0 + 1.5 * np.arange(24))], axis=1)
    body["ds"] = np.ones(len(body["X0"]))
    ok = ibl.from_workload(cfg)
    ok.ibl_step(1)
    ok.ibl_sync()


@pytest.mark.parametrize("overlap", [0, 1])
def test_sixteen_block_cluster(ibl, overlap):
    """2 x 304 markers, the sixteen-block size, alone and beside the bulk collide."""
    cfg = _wings(9.0, False)
    assert sum(len(b["X0"]) for b in cfg["bodies"]) == 608
    a, b = ibl.from_workload(cfg), ibl.from_workload(cfg)
    b.ibl_solver_preconditioner(0, -1)
    sim = oracle_from_workload(cfg)
    for c in (a, b):
        c.ibl_set_overlap(overlap)
        c.ibl_step(8)
    sim.step(8)
    compare_fields(a, sim, ibl, TOL_FIELD_FP64)
    assert rel_err(a.ibl_get_field(ibl.IBL_FIELD_U), b.ibl_get_field(ibl.IBL_FIELD_U)) < TOL_FIELD_FP64
    again = ibl.from_workload(cfg)
    again.ibl_set_overlap(1 - overlap)
    again.ibl_step(8)
    assert np.array_equal(again.ibl_get_populations(), a.ibl_get_populations())


@pytest.mark.parametrize("chord", [4.0, 7.9])
def test_rows_read_from_l2(ibl, chord):
    """Preconditioner rows kept on chip and read from L2 give the same bits, with the automatic kind too."""
    cfg = _wings(chord, True)
    runs = []
    for resident in (-1, 0):
        ctx = ibl.from_workload(cfg)
        ctx.ibl_solver_preconditioner(-1, resident)
        ctx.ibl_step(10)
        runs.append(ctx.ibl_get_populations())
    assert np.array_equal(runs[0], runs[1])
