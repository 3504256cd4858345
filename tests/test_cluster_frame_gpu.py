"""The ghost frame after steps that run in one cluster launch: cells behind periodic links are
copies of the state, corners included, isothermal ghost cells hold the wall's values - the same
bits as after one-step launches (WLBM_OPT_TILE_LOOP), whose wall pass has written both buffers of
every direction by then - and a checkpoint carries them."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
P, I, A = W.PERIODIC, W.ISOTHERMAL, W.ADIABATIC_DIFFUSE
WALLS = {"periodic": (P, P, P, P), "film": (I, I, A, A), "channel": (I, I, P, P),
         "square": (I, I, I, I), "pipe": (P, P, I, I), "duct": (P, P, A, I)}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _run(nx, ny, q, bc, storage, loop):
    import paper_1911_00180_gb300 as wl
    h = wl.WormLBM(nx, ny, q, mfp=6.0, bc=bc, t_wall=(301.0, 299.5, 300.5, 300.0), storage=storage)
    h.wlbm_set_option(wl.wlbm.OPT_TILE_LOOP, loop)
    h.wlbm_init_temperature(W.random_dT(nx, ny, 3))
    h.wlbm_step(2)
    h.wlbm_step(9)
    out = h.wlbm_get_state().cpu().numpy()
    blob = h.wlbm_save()
    h.close()
    g = wl.WormLBM(nx, ny, q, mfp=6.0, bc=bc, t_wall=(301.0, 299.5, 300.5, 300.0), storage=storage)
    g.wlbm_load(blob)
    assert np.array_equal(g.wlbm_get_state().cpu().numpy(), out)
    g.close()
    return out


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("walls", list(WALLS))
@pytest.mark.parametrize("nx,ny,q", [(2, 1, 8), (37, 53, 24), (96, 11, 64)])
def test_frame(nx, ny, q, walls, storage):
    bc = WALLS[walls]
    s = _run(nx, ny, q, bc, storage, 0)
    one = _run(nx, ny, q, bc, storage, 1)
    if bc[0] == P:
        assert np.array_equal(s[:, :, 0], s[:, :, -2]) and np.array_equal(s[:, :, -1], s[:, :, 1])
    if bc[2] == P:
        assert np.array_equal(s[:, 0], s[:, -2]) and np.array_equal(s[:, -1], s[:, 1])
    for side, cells in enumerate((np.s_[:, 1:-1, 0], np.s_[:, 1:-1, -1], np.s_[:, 0, 1:-1],
                                  np.s_[:, -1, 1:-1])):
        if bc[side] == I:
            assert np.array_equal(s[cells], one[cells]), side
            assert np.all(s[cells].max(axis=1) == s[cells].min(axis=1))
    assert np.array_equal(s[:, 1:-1, 1:-1], one[:, 1:-1, 1:-1])
