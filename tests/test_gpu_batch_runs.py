"""The runs of tiles that a block of the batch draws at a time, by the work there
is: with one block per SM four small beds (110 to 250 tiles) take single draws or
runs of two and eight beds runs of four, at ragged run ends.

Bars: every field bit for bit equal to single-domain stepping.  A batch whose
tiles are all resident at once takes about one tile's time a step, whatever
their number: less than 2.5 times a batch of one tile (runs of four tiles would
take four tiles' time)."""
import time

import numpy as np
import pytest

from paper_2310_17214_gb300 import inputs as I
from paper_2310_17214_gb300._native import Batch, Domain

pytestmark = pytest.mark.gpu


def make(p, precision="fp32"):
    phi = I.disc_phi(p["nx"], p["ny"], p["nx"] / 2, p["ny"] / 2, p["ny"] / 5, 4.0).reshape(-1)
    d = Domain(p, precision)
    d.set_phase_field(phi)
    d.set_fields((1 - phi) * 300.0 + phi * 600.0)
    return d


@pytest.mark.parametrize("n", [2, 4, 8])
@pytest.mark.parametrize("tile", ["32x8", "32x16", "64x4"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_runs_equal_one_by_one(precision, tile, n):
    probs = I.config5(n=n, seed=9, precision=precision, base=(64, 32))
    single, batched = [make(p, precision) for p in probs], [make(p, precision) for p in probs]
    b = Batch(batched)
    b.set_config(tile, 1)
    b.step(7)
    for d, e in zip(single, batched):
        d.step(7)
        x, y = d.get("T", "g", "u"), e.get("T", "g", "u")
        for k in x:
            assert np.array_equal(x[k], y[k]), k
        assert e.scalars()["step"] == 7
    b.close()
    for d in single + batched:
        d.close()


def us_per_step(probs):
    import torch
    doms = [make(p) for p in probs]
    b = Batch(doms)
    best = np.inf
    for _ in range(6):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        b.step(200)
        torch.cuda.synchronize()
        best = min(best, (time.perf_counter() - t0) / 200 * 1e6)
    b.close()
    for d in doms:
        d.close()
    return best


def test_a_resident_batch_takes_one_tiles_time():
    one = dict(I.config5(n=1, base=(64, 32))[0], nx=32, ny=8)
    few = us_per_step(I.config5(n=5, base=(64, 32)))
    assert few < 2.5 * us_per_step([one]), few
