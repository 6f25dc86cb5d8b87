"""The Newton T recovery of a loaded state over warm starts: the one-step form
(close starts) and the iterations (distant ones) against the oracle's iterations
from the same start, for 1, 3 and 9 species. (Not against the temperature the
state was made from: above 6000 K the fits of the 9 species turn over and the
energy has a second root, which both reach from 18000 K.)

Bar: 2e-13. F and H are sums of terms up to about 30 Cv T (formation
enthalpies), each good to a few 2^-53, in the oracle's state and in the recovery."""
import numpy as np
import pytest

import oracle as orc
from paper_2504_13750_gb300 import inputs

pytestmark = pytest.mark.gpu

STARTS = [1.0, 1.0 + 1e-12, 1.0 - 1e-7, 1.0001, 0.99, 1.05, 0.8, 1.5, 0.45, 3.0]
TEMPS = [250.0, 300.0, 999.0, 1000.5, 2300.0, 4100.0, 6000.0]


@pytest.mark.parametrize("scale", [1.0, 1e-9, 1e9])
@pytest.mark.parametrize("name", ["h2air_synth", "global_h2o2_g129", "ideal_gamma14"])
def test_recovery_over_warm_starts(name, scale):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_13750_gb300 import build, janc

    build.build()
    mech = inputs.load_mechanism(name)
    ny, nx, ns = len(TEMPS), len(STARTS), mech["ns"]
    T = np.repeat(np.array(TEMPS)[:, None], nx, axis=1)
    w = np.arange(1, ns + 1, dtype=np.float64)
    Y = np.ascontiguousarray(np.broadcast_to((w / w.sum())[:, None, None], (ns, ny, nx)))
    p = np.full((ny, nx), scale * inputs.ATM)
    U = orc.prim_to_cons(mech, T, p, np.full((ny, nx), 300.0), np.full((ny, nx), -40.0), Y)
    g = janc.Grid(mech, nx, ny, 1e-3, 1e-3, [1, 1, 1, 1], chemistry=False)
    T0 = T * np.array(STARTS)[None, :]
    g.set_state(U, T0)
    Tg = g.get_state()[1]
    assert g.status()["status"] == 0
    g.close()
    To = orc.newton(mech, inputs.grid_dict(nx, ny, 1e-3, 1e-3, [1, 1, 1, 1]), U, T0)
    To = np.asarray(To[0] if isinstance(To, tuple) else To).reshape(T.shape)
    assert np.max(np.abs(Tg - To) / To) < 2e-13


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e300])
@pytest.mark.parametrize("name", ["h2air_synth", "global_h2o2_g129", "ideal_gamma14"])
def test_recovery_refuses_starts_that_are_no_temperature(name, bad):
    """A warm start that is not finite raises a status bit in its cell, as the
    iterations from it end (NaN is no root); the good cells beside it are as without
    it. 1e300 K does so for 9 species (its 5th power overflows); with constant heat
    capacities one iteration leads back to the root."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_13750_gb300 import build, janc

    build.build()
    mech = inputs.load_mechanism(name)
    ny, nx, ns = 3, 40, mech["ns"]
    T = np.random.default_rng(5).uniform(300.0, 2300.0, (ny, nx))
    w = np.arange(1, ns + 1, dtype=np.float64)
    Y = np.ascontiguousarray(np.broadcast_to((w / w.sum())[:, None, None], (ns, ny, nx)))
    z = np.zeros((ny, nx))
    U = orc.prim_to_cons(mech, T, np.full((ny, nx), inputs.ATM), z, z, Y)
    g = janc.Grid(mech, nx, ny, 1e-3, 1e-3, [1, 1, 1, 1], chemistry=False)
    g.set_state(U, T)
    want = g.get_state()[1]
    assert g.status()["status"] == 0
    T0 = T.copy()
    T0[1, 17] = bad
    g.set_state(U, T0)
    got, st = np.empty_like(T), g.status()["status"]
    janc.janc_get_state(g.handle, np.empty_like(U), got, check=False)
    g.close()
    good = np.ones(T.shape, bool)
    good[1, 17] = False
    assert np.array_equal(got[good], want[good])
    if np.isfinite(bad) and ns < 9:
        assert st == 0 and abs(got[1, 17] / want[1, 17] - 1.0) < 2e-13
    else:
        assert st & (janc.ST_NONFINITE | janc.ST_NEWTON_FAIL | janc.ST_NONPOSITIVE)
