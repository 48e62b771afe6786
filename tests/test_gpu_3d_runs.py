"""The 3-D FP64 / FP32 schedules by the planes a resident block has to do (one
block per SM in FP64, three in FP32; 152 SMs): runs that shrink from sixteen planes
(16 to 32 planes a block) and from 32 (beyond), ragged in every direction, and
closed domains under them, whose P0 is set in the launch by the last of the
runs to arrive.

Bars: against the equal runs of the z-march bit for bit at fixed P0; against the
oracle, the suite's FP64 1e-10."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2310_17214_gb300 import inputs as I
from paper_2310_17214_gb300._native import Domain

pytestmark = pytest.mark.gpu


def problem(nx, ny, nz, bc):
    p = I._base(3, nx, ny, nz)
    I.lattice_air(p, 0.05)
    p.update(bc=bc, A_u=60.0, A_T=50.0, eta=2.5, inlet_parabolic=1, u_in=0.02, Ts_uniform=480.0,
             wall_T=[0, 0, 420.0, 0, 0, 0], p0_mode="fixed" if bc[0] == "inlet" else "closed")
    return p, I.random_state(p, 7, T_range=(300.0, 450.0), u_amp=0.01)


def domain(p, f, precision, kernel=None):
    d = Domain(p, precision)
    d.set_phase_field(f["phi"])
    d.set_fields(f["T"], None, f["u"])
    if kernel:
        d.select_kernel(kernel)
    return d


# FP64: 2,880 and 5,712 tile-planes (from sixteen, from 32); FP32: 7,350 and 15,104
@pytest.mark.parametrize("precision,shape", [("fp64", (128, 96, 60)), ("fp64", (201, 121, 51)),
                                             ("fp32", (201, 119, 70)), ("fp32", (251, 123, 118))])
def test_default_schedule_equals_the_march(precision, shape):
    p, f = problem(*shape, ["inlet", "outlet", "wall", "wall", "periodic", "periodic"])
    out = []
    for kernel in (None, "march"):
        d = domain(p, f, precision, kernel)
        d.step(3)
        out.append(d.get("T", "g", "u", "rho"))
        d.close()
    for k, a in out[0].items():
        assert np.all(np.isfinite(a)), k
        assert np.array_equal(a, out[1][k]), k


@pytest.mark.parametrize("bc", [["periodic"] * 6, ["periodic"] * 2 + ["wall"] * 2 + ["periodic"] * 2])
def test_closed_domain_under_shrinking_runs(bc):
    """37 x 19 x 41 closed: runs of sixteen, eight and four planes, the last one cut."""
    p, f = problem(37, 19, 41, bc)
    ora = O.OracleState(p, f["phi"], f["T"], u=f["u"])
    ora.step(25)
    u, rho, ph = ora.moments()
    d = domain(p, f, "fp64", "tiled")
    d.step(25)
    got, sc = d.get("T", "g", "u", "rho", "Ph"), d.scalars()
    d.close()
    ref = {"T": ora.T, "g": ora.g.reshape(ora.Q, ora.N), "u": u, "rho": rho, "Ph": ph}
    for k, r in ref.items():
        a, b = np.asarray(got[k]).reshape(-1), np.asarray(r).reshape(-1)
        assert np.max(np.abs(a - b)) <= 1e-10 * np.max(np.abs(b)), k
    assert sc["step"] == 25 and abs(sc["P0"] / ora.P0 - 1) <= 1e-10
    assert abs(sc["I"] / ora.scal[3] - 1) <= 1e-10
