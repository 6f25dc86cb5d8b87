"""The forms that only larger grids select, by the number of cells (the sizes
here cross the thresholds at 152 SMs): face tiles of 8, 16 and 32 faces with
and without derivatives for 4, 6 and 12 variables, the adjoint's cell pass in
blocks of 2 and 4 rows, its 16-face tiles, the chemistry and its VJP in their
large-grid blocks, and the AMR kernels in blocks of 128 and 256 threads with one
thread a line. References and bars are those of the same checks on small grids
(test_gpu_tiles.py, test_gpu_adjoint.py, test_gpu_amr.py)."""
import numpy as np
import pytest

import oracle as orc
from paper_2504_13750_gb300 import inputs

pytestmark = pytest.mark.gpu

MECHS = {k: inputs.load_mechanism(k) for k in ("h2air_synth", "global_h2o2_g129", "ideal_gamma14")}


@pytest.fixture(scope="module")
def J():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2504_13750_gb300 import build, janc

    build.build()
    return janc


def _state(mech, nx, ny, seed, bc):
    """A tube with noise in T and both velocities (a unique arg-max of the LF speeds)."""
    Y = {9: None, 3: np.array([0.1, 0.8, 0.1]), 1: np.ones(1)}[mech["ns"]]
    st = inputs.tube(mech, nx, ny, perturb_seed=seed, Y=Y)
    rng = np.random.default_rng(seed)
    st["T"] = st["T"] + rng.normal(0.0, 5.0, (ny, nx))
    st["u"] = rng.normal(0.0, 60.0, (ny, nx))
    st["v"] = rng.normal(0.0, 60.0, (ny, nx))
    st["grid"]["bc"] = list(bc)
    return st, orc.prim_to_cons(mech, st["T"], st["p"], st["u"], st["v"], st["Y"])


@pytest.mark.parametrize("name", ["ideal_gamma14", "global_h2o2_g129"])
def test_tiles_of_32_faces(J, name):
    mech = MECHS[name]
    st, U = _state(mech, 1301, 403, 2, (0, 1, 2, 2))
    g = J.Grid.from_grid_dict(mech, st["grid"], chemistry=False)
    g.set_state(U, st["T"])
    _, Fx, Gy, _ = g.rhs()
    g.close()
    _, Fx0, Gy0, _ = orc.rhs(mech, st["grid"], U, st["T"])
    for a, b in ((Fx, Fx0), (Gy, Gy0)):
        for k in range(mech["ns"] + 3):
            assert np.max(np.abs(a[k] - np.asarray(b)[k])) <= 1e-12 * np.max(np.abs(np.asarray(b)[k]))


@pytest.mark.parametrize("store", [False, True], ids=["recompute", "store_faces"])
@pytest.mark.parametrize("name,chem,nx,ny", [
    ("h2air_synth", 1, 150, 80), ("h2air_synth", 1, 400, 130), ("h2air_synth", 1, 700, 130), ("h2air_synth", 1, 1210, 140),
    ("global_h2o2_g129", 3, 150, 80), ("global_h2o2_g129", 3, 400, 130), ("global_h2o2_g129", 3, 1301, 240),
    ("ideal_gamma14", 0, 400, 130), ("ideal_gamma14", 0, 700, 130), ("ideal_gamma14", 0, 1301, 370)])
def test_trajectory_dot_product(J, name, chem, nx, ny, store):
    """Two steps in two segments: <seed, dU^N> of the oracle's tangent against
    <dL/dU^0, dU^0> of the reverse sweep, and the forward's bits against janc_step."""
    mech = MECHS[name]
    st, U = _state(mech, nx, ny, 6, (0, 1, 2, 2))
    dt, n = 4e-9, 2
    g = J.Grid.from_grid_dict(mech, st["grid"], chemistry=chem)
    J.janc_set_adjoint_mode(g.handle, J.ADJ_STORE_FACES if store else J.ADJ_RECOMPUTE)
    g.set_state(U, st["T"])
    g.step(n, dt=dt)
    Us, Ts = g.get_state()
    g.set_state(U, st["T"])
    rng = np.random.default_rng(7)
    scale = np.maximum(np.abs(U).reshape(U.shape[0], -1).max(axis=1), 1e-12)[:, None, None]
    seed = rng.normal(size=U.shape) / scale
    gU0 = np.zeros_like(U)
    J.janc_step_adjoint(g.handle, n, dt, 1, J.LOSS_SEEDED, seed, gU0)
    UN, TN = g.get_state()
    g.close()
    assert np.array_equal(UN, Us) and np.array_equal(TN, Ts)
    V = rng.normal(size=(2,) + U.shape) * (1e-3 * scale)
    orc.set_threads(0)
    dUN, _, _, s = orc.trajectory_tangent(mech, st["grid"], U, st["T"], V, n, dt, chem=orc.CHEM_EXPLICIT if chem == 3 else bool(chem))
    assert s == 0
    for l in range(2):
        a, b = float(np.sum(seed * dUN[l])), float(np.sum(gU0 * V[l]))
        assert abs(a - b) <= 1e-8 * np.sum(np.abs(seed * dUN[l])), (l, a, b)


@pytest.mark.parametrize("nx,ny", [(384, 64), (512, 80)])
def test_full_layer_of_many_blocks(J, nx, ny):
    """Every block of layer 1 present (384 and 640 of them): the layer steps like
    the undivided fine grid with dt / 2, to 1e-11 a step."""
    mech = MECHS["h2air_synth"]
    st = inputs.tube(mech, nx, ny, perturb_seed=3)
    a = J.Amr(mech, st["grid"], chemistry=True, levels=1, threshold=-1.0, n_buffer=0, regrid_every=1000)
    a.set_primitive(st["T"], st["p"], st["u"], st["v"], np.ascontiguousarray(st["Y"]))
    U0, T0 = a.base()
    gf = dict(st["grid"], nx=2 * nx, ny=2 * ny, dx=st["grid"]["dx"] / 2, dy=st["grid"]["dy"] / 2)
    f = J.Grid.from_grid_dict(mech, gf)
    f.set_state(np.ascontiguousarray(np.repeat(np.repeat(U0, 2, 1), 2, 2)), np.ascontiguousarray(np.repeat(np.repeat(T0, 2, 0), 2, 1)))
    dt = 8e-9
    a.step(2, dt=dt)
    f.step(4, dt=dt / 2)
    pos, UL, TL = a.layer(1)
    assert len(pos) == nx * ny // 64 and a.status() == 0
    Ug, Tg = np.zeros((UL.shape[1], 2 * ny, 2 * nx)), np.zeros((2 * ny, 2 * nx))
    for k, (bx, by) in enumerate(pos):
        Ug[:, by * 16:(by + 1) * 16, bx * 16:(bx + 1) * 16] = UL[k]
        Tg[by * 16:(by + 1) * 16, bx * 16:(bx + 1) * 16] = TL[k]
    Uf, Tf = f.get_state()
    a.close()
    f.close()
    for k in range(Ug.shape[0]):
        assert np.max(np.abs(Ug[k] - Uf[k])) <= 2e-11 * np.max(np.abs(Uf[k]))
    assert np.max(np.abs(Tg - Tf) / Tf) < 2e-11
