"""The implicit integrator at every reaction count it is compiled for (0 to 4;
each count solves a system of its own size), with the reaction orders and the
reversible form it treats apart, cell by cell against the oracle's full
(K + 1)-unknown Newton.

Bars: both sides stop at an update below 1e-13 (species absolute, temperature
relative to the start) in each of at most 64 sub-steps, so FP64 increments agree
to 64 x 1e-13 of that scale; FP32 domains to the bar of their fallback
integrator.  Cells on which the oracle itself does not converge are left out."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2310_17214_gb300 import inputs as I
from paper_2310_17214_gb300._native import Domain

pytestmark = pytest.mark.gpu

EXTRA = [  # fractional orders and a temperature exponent; second order
    {"A": 2e7, "b": 0.25, "EaR": 14000.0, "order": [0.7, 1.3, 0, 0, 0, 0],
     "stoich": [-1, -2, 0, 1, 2, 0]},
    {"A": 3e7, "b": 0.0, "EaR": 13000.0, "order": [0, 0, 2, 0, 0, 0],
     "stoich": [0, -0.5, -1, 1, 0, 0]}]


@pytest.mark.parametrize("J", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_increments_at_every_reaction_count(J, precision):
    p = I.config4(nx=24, ny=9, precision=precision)
    p["reactions"] = (I.two_step_mechanism() + EXTRA)[:J]
    rng = np.random.default_rng(J)
    N = 24 * 9
    M = np.asarray(p["M"])
    Yin = np.asarray(p["Y_in"])
    e1 = rng.uniform(0, 1, N) * Yin[0] / M[0]
    e2 = rng.uniform(0, 1, N) * e1
    s = np.array([r["stoich"] for r in I.two_step_mechanism()])
    Y = Yin[:, None] + M[:, None] * (s[0][:, None] * e1 + s[1][:, None] * e2)
    Y[0, :5] = 0.0   # no fuel
    Y[1, 5:9] = -1e-9  # an undershoot of the transport
    T = rng.uniform(300.0, 2100.0, N)
    d = Domain(p, precision)
    d.set_phase_field(np.zeros(N), np.full(N, 300.0))
    d.set_fields(T, Y.reshape(-1))
    dY, dT = d.chem_increments()
    g = d.get("T", "Y")
    P0 = d.scalars()["P0"]
    d.close()
    moved, compared = 0.0, 0
    for c in range(N):
        Tc, Yc = float(g["T"][c]), g["Y"][:, c].astype(np.float64)
        rho = P0 / (I.R_GAS * Tc * np.sum(Yc / M)) / p["rho_ref"]
        ry, rt, rc = O.chem_implicit(p, Tc, Yc, rho)
        if rc != 0:
            continue
        compared += 1
        moved = max(moved, abs(rt))
        if precision == "fp64":
            assert np.max(np.abs(dY[:, c] - ry)) <= 6.4e-12, c
            assert abs(dT[c] - rt) <= 6.4e-12 * Tc, c
        else:
            assert np.all(np.abs(dY[:, c] - ry) <= 1e-4 * np.abs(ry) + 4e-6 * np.abs(Yc) + 1e-12), c
            assert abs(dT[c] - rt) <= 1e-4 * abs(rt) + 4e-6 * Tc, c
    assert (moved > 0.1) == (J > 0) and compared >= N - 2
