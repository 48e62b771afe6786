"""The reduction scalars of domains whose last step's sums are combined by the
first block of the next launch (fixed P0).

One plane: a 24 x 160 x 1 lattice has 20 tile-planes of 32 x 8 cells and 40
partial slots, fewer planes than the resident grid of the z-march.

Reading the scalars combines the last step's sums at once instead of in the next
launch: to the same bits, under every block size of the step (FP64 tiles of 2,
4 and 8 rows, the z-march) and beside more than one share of 256 slots.

Bars: the suite's, FP64 1e-10 and FP32 1e-4 relative to the oracle's scalars; the
moment of reading moves no bit."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2310_17214_gb300 import inputs as I
from paper_2310_17214_gb300._native import Domain

pytestmark = pytest.mark.gpu


def problem(dim, nx, ny, nz):
    p = I._base(dim, nx, ny, nz)
    I.lattice_air(p, 0.05)
    p.update(bc=["inlet", "outlet", "wall", "wall", "periodic", "periodic"], A_u=60.0, A_T=50.0,
             eta=2.5, inlet_parabolic=1, u_in=0.02, Ts_uniform=480.0, p0_mode="fixed")
    return p, I.random_state(p, 7, T_range=(300.0, 450.0), u_amp=0.01)


def domain(p, f, precision, kernel=None):
    d = Domain(p, precision)
    d.set_phase_field(f["phi"])
    d.set_fields(f["T"], None, f["u"])
    if kernel:
        d.select_kernel(kernel)
    return d


@pytest.mark.parametrize("kernel", [None, "tiled", "march", "march_prefetch"])
@pytest.mark.parametrize("precision,bar", [("fp64", 1e-10), ("fp32", 1e-4)])
def test_one_plane_scalars_match_oracle(precision, bar, kernel):
    p, f = problem(3, 24, 160, 1)
    ora = O.OracleState(p, f["phi"], f["T"], u=f["u"])
    d = domain(p, f, precision, kernel)
    for n in (1, 7, 8):
        ora.step(n)
        d.step(n)
        sc, dg = d.scalars(), d.diagnostics()
        got = [sc["I"], sc["flux_in"], sc["flux_out"], dg["flux_in_total"], dg["flux_out_total"]]
        ref = [ora.scal[3], ora.scal[4], ora.scal[5], ora.scal[7], ora.scal[8]]
        assert all(r != 0.0 for r in ref)
        assert np.all(np.abs(np.subtract(got, ref)) <= bar * np.abs(ref)), (n, got, ref)
    d.close()


@pytest.mark.parametrize("shape", [(2, 128, 64, 1), (2, 300, 120, 1), (2, 600, 500, 1),
                                   (3, 40, 24, 20)])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_fp16"])
def test_reading_the_scalars_moves_no_bit(precision, shape):
    p, f = problem(*shape)
    seen = []
    for read in (False, True):
        d = domain(p, f, precision)
        for _ in range(20):
            d.step(1)
            if read:
                d.scalars()
        dg = d.diagnostics()
        seen.append((d.scalars(), dg["flux_in_total"], dg["flux_out_total"]))
        d.close()
    assert seen[0] == seen[1]
