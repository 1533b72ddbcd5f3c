"""GPU stencils of coordinates that lie a rounding residue beside a node: the
first node and the weights (Eq. 14) must come from the same floor."""
import numpy as np
import pytest

import workloads as W
from tests.parity import TOL_FIELD_FP64, compare_fields, oracle_from_workload
from tests.test_gpu_points import _dev, _oracle_moments, _pair

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# beside 0, and on both sides of 2^-64, the resolution of the integer split
RESIDUES = [-1e-20, -1e-30, -5e-324, -2.0 ** -64, -2.0 ** -65, -1e-19, -1e-17, -0.0, 5e-324, 1e-20, 1e-17]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("q,shape", [(19, (13, 11, 21)), (9, (1, 23, 37))])
def test_points_beside_node_zero(ibl, q, shape, prec):
    """A stencil moves by the residue: values at most 1e-17 times the fields'
    differences away from those at 0, so the same to 1e-14."""
    ctx, sim = _pair(ibl, q, prec, shape, [W.PERIODIC] * 6, 2)
    d = sim.lat.d
    X = []
    for a in range(d):
        for r in RESIDUES:
            x = [7.25, 6.5, 5.75]
            x[a] = r
            X.append(x)
    at0 = np.where(np.abs(np.array(X)) < 1e-10, 0.0, np.array(X))
    U, rho = ctx.ibl_interpolate_points(_dev(X))
    U0, rho0 = ctx.ibl_interpolate_points(_dev(at0))
    assert (U - U0).abs().max() < 1e-14 and (rho - rho0).abs().max() < 1e-14
    V, ds = np.full((len(X), d), 0.03), np.ones(len(X))
    out, out0 = (ctx.ibl_spread_points(_dev(x), _dev(V), _dev(ds)) for x in (X, at0))
    assert (out - out0).abs().max() < len(X) * 2 * 2.0 ** -46
    # at node 0 itself: 1/4, 1/2, 1/4 on that axis, against the oracle's fields
    lat_rho, _ = _oracle_moments(sim)
    r = lat_rho[:, :, [-1, 0, 1]] @ np.array([0.25, 0.5, 0.25])
    cx = 0.25 * (1 + np.cos(0.5 * np.pi * np.arange(-1.5, 2.0)))
    cz = 0.25 * (1 + np.cos(0.5 * np.pi * (np.arange(-1, 3) - 0.75)))
    want = np.einsum("zy,z,y->", r[4:8, 5:9], cz, cx) if d == 3 else r[0, 5:9] @ cx
    assert abs(rho[0].item() - want) < (1e-10 if prec == "fp64" else 1e-5)


@pytest.mark.parametrize("residue", [-1e-20, -5e-324, -1e-19])
def test_marker_beside_node_zero(ibl, residue):
    """A marker a residue below a periodic face: the run of the one on it."""
    still = {"kind": W.WAVE_CONST, "amp": 0.0, "offset": 0.0}
    body = {"X0": np.array([[residue, 0.0]]), "ds": np.ones(1), "hinge": (0, 0, 0), "axis": (0, 0, 1),
            "origin": (0.0, 12.4, 0.0), "A": still, "alpha": still, "beta": 0.0, "phi": 0.0, "f": 1 / 300.0, "J": 0.0}
    cfg = {"lattice": 9, "tau": 0.8, "grid": W.grid(24, 28, 1, [W.PERIODIC] * 6, precision="fp64"), "bodies": [body],
           "u0": (0.03, 0.01, 0.0), "reference": {"U_ref": 0.1, "L": 1.0, "rho_ref": 1.0}}
    at0 = dict(cfg, bodies=[dict(body, X0=np.zeros((1, 2)))])
    ctx, sim = ibl.from_workload(cfg), oracle_from_workload(at0)
    ctx.ibl_step(5)
    sim.step(5)
    compare_fields(ctx, sim, ibl, TOL_FIELD_FP64)
