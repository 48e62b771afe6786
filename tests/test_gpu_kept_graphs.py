"""A domain keeps the graph of its step pairs from one long call to the next.
Whatever changes between the calls (the kernel, the starting parity, the state,
the surrogate), the run must equal single-step calls bit for bit."""
import numpy as np
import pytest

from paper_2310_17214_gb300 import inputs as I
from paper_2310_17214_gb300 import surrogate as S
from paper_2310_17214_gb300._native import Domain, Mlp, MLP_PARAMS

pytestmark = pytest.mark.gpu


def _run(p, f, precision, script, long_calls):
    d = Domain(p, precision)
    d.set_phase_field(f["phi"])
    d.set_fields(f["T"], f["Y"])
    for kernel, n in script:
        if kernel == "state":
            d.set_fields(f["T"], f["Y"])
        elif kernel:
            d.select_kernel(kernel)
        for k in ([n] if long_calls else [1] * n):
            d.step(k)
    out, sc = d.get("T", "Y", "u", "g"), d.scalars()
    d.close()
    return out, sc


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_fp16"])
def test_kept_graphs_follow_changes_between_calls(precision):
    p = I.config6(nx=96, ny=32, precision=precision)
    f = I.config6_fields(p)
    script = [(None, 40), (None, 41), ("persistent", 40), ("tiled", 33), ("state", 40), (None, 40)]
    a, sa = _run(p, f, precision, script, True)
    b, sb = _run(p, f, precision, script, False)
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    for k in ("P0", "step", "u_in", "fuel"):
        assert sa[k] == sb[k], k


def test_kept_graphs_follow_a_new_surrogate():
    p = I.config4(nx=128, ny=40, precision="fp32", chem="surrogate")
    p["bed"] = {"count": 4, "amin": 5, "amax": 8, "porosity": 0.6, "x0": 64}
    p["ignite"] = [8, 40, 1800.0]
    f = I.config4_fields(p)
    X = np.array([[300.0] + list(p["Y_in"]) + [p["P0"]]] * 2)
    X[1, 0] = 2500.0
    stats = (X.mean(axis=0), X.std(axis=0), np.zeros(6), np.zeros(6))
    out = []
    for long_calls in (True, False):
        d = Domain(p, "fp32")
        d.set_phase_field(f["phi"], f["Ts"])
        d.set_fields(f["T"], f["Y"])
        nets = [Mlp(), Mlp()]
        for net, tol in zip(nets, (-1.0, 1e30)):  # every cell falls back; every cell accepted
            net.set_params(np.zeros(MLP_PARAMS, dtype=np.float32))
            d.set_surrogate(net, S.make_surrogate(stats, X, 0.0, p["species"], tol))
            for k in ([40] if long_calls else [1] * 40):
                d.step(k)
        out.append(d.get("T", "Y", "g"))
        d.close()
        for net in nets:
            net.close()
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]), k
