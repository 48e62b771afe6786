"""The runs of planes of the FP16-stored 3-D step against the z-march, which cuts
the same planes into other runs: every field bit for bit after three steps, on
a lattice of less than a tile and few planes (runs of one plane), ragged tiles
in runs that fit one wave, and two long enough for the runs that shrink from
eight and from sixteen planes, whose last run is cut short."""
import numpy as np
import pytest

from paper_2310_17214_gb300 import inputs as I
from paper_2310_17214_gb300._native import Domain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(19, 7, 5), (70, 43, 53), (201, 121, 51), (201, 121, 90)])
@pytest.mark.parametrize("zbc", ["periodic", "wall"])
def test_half_runs_equal_the_march(nx, ny, nz, zbc):
    p = I._base(3, nx, ny, nz)
    I.lattice_air(p, 0.05)
    p.update(bc=["inlet", "outlet", "periodic", "periodic", zbc, zbc], A_u=60.0, A_T=50.0, eta=2.5,
             inlet_parabolic=0, u_in=0.02, Ts_uniform=480.0, p0_mode="fixed")
    f = I.random_state(p, 7, T_range=(300.0, 450.0), u_amp=0.01)
    out = {}
    for kern in ("tiled", "march"):
        d = Domain(p, "fp32_fp16")
        d.set_phase_field(f["phi"])
        d.set_fields(f["T"], None, f["u"])
        d.select_kernel(kern)
        d.step(3)
        out[kern] = d.get("T", "g", "u", "rho")
        d.close()
    for k, a in out["tiled"].items():
        assert np.all(np.isfinite(a)), k
        assert np.array_equal(a, out["march"][k]), k
