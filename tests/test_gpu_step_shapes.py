"""Shapes at which the step kernels can go wrong: pairs of cells on odd rows,
ragged tiles, every height of the FP64 tile, runs of planes of the 3-D
schedule, and caller arrays that do not start on a pair boundary.

Bars: FP64 max relative error 1e-10 and FP32 L2 relative error 1e-4 against
the oracle (the suite's bars); different block schedules of the same update
bit for bit."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2310_17214_gb300 import inputs as I
from paper_2310_17214_gb300._native import Domain, step_noalloc

pytestmark = pytest.mark.gpu

WALLS = ["inlet", "outlet", "wall", "wall", "periodic", "periodic"]
BOX = ["periodic"] * 6


def problem(dim, nx, ny, nz, bc):
    p = I._base(dim, nx, ny, nz)
    I.lattice_air(p, 0.05)
    p.update(bc=bc, A_u=60.0, A_T=50.0, eta=2.5, inlet_parabolic=1, u_in=0.02, Ts_uniform=480.0,
             wall_T=[0, 0, 420.0, 0, 0, 0], p0_mode="closed" if bc is BOX else "fixed")
    return p, I.random_state(p, 7, T_range=(300.0, 450.0), u_amp=0.01)


def run(p, f, precision, kernel, steps):
    d = Domain(p, precision)
    d.set_phase_field(f["phi"])
    d.set_fields(f["T"], None, f["u"])
    if kernel:
        d.select_kernel(kernel)
    d.step(steps)
    out = d.get("T", "g", "u")
    d.close()
    return out


# 2-D: one pair, odd rows, one row, rows beyond the tile; (33, 3), (640, 11) and
# (1300, 100) take FP64 tiles of 2, 4 and 8 rows on 152 SMs
@pytest.mark.parametrize("bc", [WALLS, BOX])
@pytest.mark.parametrize("nx,ny", [(2, 4), (33, 3), (35, 9), (64, 17), (640, 11), (1300, 100)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_2d_shapes_against_oracle(nx, ny, bc, precision):
    p, f = problem(2, nx, ny, 1, bc)
    ora = O.OracleState(p, f["phi"], f["T"], u=f["u"])
    ora.step(12)
    u, _, _ = ora.moments()
    got = run(p, f, precision, None, 12)
    ref = {"T": ora.T, "g": ora.g.reshape(ora.Q, ora.N), "u": u}
    for k in ref:
        a, b = np.asarray(got[k]), np.asarray(ref[k]).reshape(got[k].shape)
        if precision == "fp64":
            assert np.max(np.abs(a - b)) <= 1e-10 * np.max(np.abs(b)), k
        else:
            assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b), k


@pytest.mark.parametrize("nx,ny,nz", [(37, 9, 1), (34, 8, 3), (33, 17, 5), (64, 10, 37), (36, 8, 70)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_3d_schedules_cover_every_plane(nx, ny, nz, precision):
    """The shrinking runs (tiled), the equal runs (march) and the march that
    loads its populations early give the same bits on every cell."""
    p, f = problem(3, nx, ny, nz, WALLS)
    ref = run(p, f, precision, "march", 5)
    for kern in ("tiled", "march_prefetch"):
        got = run(p, f, precision, kern, 5)
        for k in ref:
            assert np.array_equal(got[k], ref[k]), (kern, k)


def test_caller_arrays_off_the_pair_boundary():
    """pflb_step_noalloc on arrays that start 4 bytes off an 8-byte boundary:
    the same bits as on aligned ones."""
    import torch
    p, f = problem(2, 40, 10, 1, WALLS)
    N = 400
    out = []
    for off in (0, 1):
        def dev(a):
            t = torch.empty(a.size + 2, dtype=torch.float32, device="cuda")[off:off + a.size]
            return t.copy_(torch.as_tensor(np.asarray(a, dtype=np.float32).reshape(-1)))
        d = Domain(p, "fp32")
        d.set_phase_field(f["phi"])
        d.set_fields(f["T"], None, f["u"])
        g0, sc = d.get("g", dtype=np.float32), d.scalars()
        d.close()
        arr = {"phi": dev(f["phi"]), "g_in": dev(g0), "T_in": dev(f["T"]),
               "g_out": dev(np.zeros(9 * N)), "T_out": dev(np.zeros(N))}
        assert arr["T_in"].data_ptr() % 8 == 4 * off
        step_noalloc(p, "fp32", arr, sc)
        torch.cuda.synchronize()
        out.append((arr["g_out"].cpu().numpy(), arr["T_out"].cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
