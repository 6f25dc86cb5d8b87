"""The rate constants of the compiled H2-air chemistry kernels (fixed-point
base-2 logarithms between 256 K and 8192 K, FP64 outside) against the oracle's
point-implicit step: one reactor per cell, at temperatures around both ends, at
powers of two and between, for ordinary, stiff and vanishing time steps, and
for a table whose numbers do not fit the fixed-point form.

Bar: a reactor's change within 1e-9 of its largest species change. The G_k as
doubles are good to 2^-48; a net rate may cancel by four orders before that."""
import numpy as np
import pytest

import oracle as orc
from paper_2504_13750_gb300 import inputs

pytestmark = pytest.mark.gpu

H2AIR = inputs.load_mechanism("h2air_synth")
TEMPS = [180.0, 255.999999, 256.0, 256.000001, 300.0, 511.9999, 512.0, 777.0, 1023.9, 1024.0, 1500.0, 2048.0, 2500.0, 4095.99,
         4096.0, 6000.0, 8191.999, 8192.0, 8300.0]


def _unfit():
    m = dict(H2AIR)
    m["Ea"] = np.array(H2AIR["Ea"], dtype=np.float64).copy()
    m["Ea"][3] = 6.0e5  # Ea / R beyond the fixed-point range
    return m


@pytest.mark.parametrize("dt", [1e-9, 1e-6, 2.0 ** -69, 2.0 ** -71])
@pytest.mark.parametrize("table", ["shipped", "unfit"])
def test_reactors_over_temperature(table, dt):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_13750_gb300 import build, janc

    build.build()
    mech = H2AIR if table == "shipped" else _unfit()
    part = {"H2": 0.02, "O2": 0.12, "H": 1e-3, "O": 5e-3, "OH": 0.02, "HO2": 1e-4, "H2O2": 1e-5, "H2O": 0.15}
    part["N2"] = 1.0 - sum(part.values())
    n = len(TEMPS)
    T = np.array(TEMPS)[None, :]
    Y = np.ascontiguousarray(np.repeat(np.asarray(inputs.premix_Y(mech, part))[:, None, None], n, axis=2))
    p, z = np.full((1, n), 5 * inputs.ATM), np.zeros((1, n))
    U0 = orc.prim_to_cons(mech, T, p, z, z, Y)
    g = janc.Grid(mech, n, 1, 1e-3, 1e-3, [1, 1, 1, 1], chemistry=True)
    g.set_state(U0, T)
    Ts = g.get_state()[1]
    assert np.max(np.abs(Ts - T) / T) < 1e-12
    janc.janc_source_step(g.handle, 1, dt)
    U = g.get_state()[0]
    assert g.status()["status"] == 0
    g.close()
    Uo, st = orc.point_implicit(mech, U0, T, dt)
    assert st == 0
    assert np.array_equal(U[:4], U0[:4])
    d, do = U[4:, 0] - U0[4:, 0], Uo[4:, 0] - U0[4:, 0]
    # the step's own change, or rounding of the stored value where that is larger
    floor = 4 * np.spacing(np.abs(U0[4:, 0])).max(axis=0)
    assert np.all(np.abs(d - do) <= np.maximum(1e-9 * np.abs(do).max(axis=0), floor))
