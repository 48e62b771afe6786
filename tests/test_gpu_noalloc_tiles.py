"""pflb_step_noalloc on a long, flat FP64 lattice: its tiles of 8 rows fit the
fixed scratch array and the lower ones that the step would take from the
occupancy alone do not (131072 x 10 cells: 8,192 tiles of 8 rows, 20,480 of 2,
16,384 slots).  The call is answered, with pflb_step's fields.

Bar: bit for bit (a cell's update does not depend on the tile)."""
import numpy as np
import pytest

from paper_2310_17214_gb300 import inputs as I
from paper_2310_17214_gb300._native import Domain, step_noalloc

pytestmark = pytest.mark.gpu


def test_noalloc_takes_a_long_flat_fp64_lattice():
    import torch
    nx, ny = 131072, 10
    p = I._base(2, nx, ny)
    I.lattice_air(p, 0.05)
    p.update(bc=["inlet", "outlet", "wall", "wall", "periodic", "periodic"], A_u=60.0, A_T=50.0,
             eta=2.5, inlet_parabolic=1, u_in=0.02, Ts_uniform=480.0, p0_mode="fixed")
    N = nx * ny
    T = np.random.default_rng(3).uniform(300.0, 450.0, N)
    d = Domain(p, "fp64")
    d.set_phase_field(np.zeros(N))
    d.set_fields(T)
    g0, sc = d.get("g"), d.scalars()
    d.step(1)
    ref = d.get("T", "g")
    d.close()
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a).reshape(-1), device="cuda")
    arr = {"phi": dev(np.zeros(N)), "T_in": dev(T), "g_in": dev(g0)}
    arr["T_out"], arr["g_out"] = torch.empty_like(arr["T_in"]), torch.empty_like(arr["g_in"])
    out = step_noalloc(p, "fp64", arr, sc)
    assert out["step"] == 1 and out["status"] == 0
    assert np.array_equal(arr["T_out"].cpu().numpy(), ref["T"])
    assert np.array_equal(arr["g_out"].cpu().numpy().reshape(ref["g"].shape), ref["g"])
