"""Face fluxes over the tile lengths that the grid size selects (4, 8, 16 and 32
faces), for 4, 6 and 12 variables, with remainders in both directions, against
the oracle. Bar: 1e-12, one right-hand side's (test_gpu_parity.py)."""
import numpy as np
import pytest

import oracle as orc
from paper_2504_13750_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(5, 4), (37, 3), (97, 33), (163, 41), (260, 70), (903, 203)])
@pytest.mark.parametrize("name", ["ideal_gamma14", "global_h2o2_g129", "h2air_synth"])
def test_tiles(name, nx, ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_13750_gb300 import build, janc

    build.build()
    mech = inputs.load_mechanism(name)
    rng = np.random.default_rng([nx, ny])
    ns = mech["ns"]
    x = np.arange(nx)[None, :] + 0.0 * np.arange(ny)[:, None]
    T = 900.0 + 700.0 * (x < nx / 2) + 5.0 * rng.standard_normal((ny, nx))
    p = inputs.ATM * (1.0 + 4.0 * (x < nx / 2)) * (1.0 + 0.01 * rng.standard_normal((ny, nx)))
    u, v = 100.0 * rng.standard_normal((ny, nx)), 50.0 * rng.standard_normal((ny, nx))
    Y = rng.uniform(0.5, 1.0, (ns, ny, nx))
    Y /= Y.sum(0)
    bc = [0, 1, 2, 2] if ny > 3 else [0, 1, 0, 1]
    grid = inputs.grid_dict(nx, ny, 1e-4, 1.3e-4, bc)
    U = orc.prim_to_cons(mech, T, p, u, v, Y)
    g = janc.Grid.from_grid_dict(mech, grid, chemistry=False)
    g.set_state(U, T)
    _, Fx, Gy, _ = g.rhs()
    g.close()
    _, Fx0, Gy0, _ = orc.rhs(mech, grid, U, T)
    for a, b in ((Fx, Fx0), (Gy, Gy0)):
        for k in range(ns + 3):
            assert np.max(np.abs(a[k] - np.asarray(b)[k])) <= 1e-12 * np.max(np.abs(np.asarray(b)[k]))
