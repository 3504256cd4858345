"""Launches that advance many steps of a small grid in one cluster's shared memory
(k_step_cluster.cu) against the one-step kernels: the arithmetic and its order are the same, so
states, moments and reductions must be equal bit for bit, for every wall set the launches
cover, bands of rows and of columns, single cells, uneven last bands and any grouping of the
steps.  WLBM_OPT_TILE_LOOP selects the one-step kernels."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
P, I, A = W.PERIODIC, W.ISOTHERMAL, W.ADIABATIC_DIFFUSE


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1911_00180_gb300  # noqa: F401


def _bits(t):
    return t.detach().cpu().contiguous().numpy().view(np.uint32)


def _run(nx, ny, q, bc, storage, parts, loop, field, speed, seed):
    import paper_1911_00180_gb300 as wl
    mfp = None
    if field:
        mfp = (2.0 + 30.0 * np.random.default_rng(seed).random((ny, nx))).astype(np.float32)
    h = wl.WormLBM(nx, ny, q, mfp=6.0, mfp_field=mfp, bc=bc, t_wall=(301.0, 299.5, 300.5, 300.0),
                   storage=storage, speed=speed)
    h.wlbm_set_option(wl.wlbm.OPT_TILE_LOOP, loop)
    h.wlbm_init_temperature(W.random_dT(nx, ny, seed))
    for n in parts:
        h.wlbm_step(n)
    h.wlbm_check()
    st = h.wlbm_get_state()
    y0 = 0 if bc[2] == A else 1
    y1 = ny + 2 if bc[3] == A else ny + 1
    out = [_bits(st[:, y0:y1, 1:-1])] + [_bits(m) for m in h.wlbm_moments()]
    out.append(np.array(h.wlbm_reduce()[:5]).view(np.uint64))
    h.close()
    return out


WALLS = {"periodic": (P, P, P, P), "film": (I, I, A, A), "channel": (I, I, P, P),
         "square": (I, I, I, I), "duct": (P, P, A, I), "tube": (P, P, A, A)}


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("walls", list(WALLS))
@pytest.mark.parametrize("nx,ny,q,parts,field,speed", [
    (2, 1, 8, (7,), False, 1.0),            # smallest grids: halos wrap onto their own cells
    (4, 2, 16, (3, 2, 1, 4), True, 1.0),
    (64, 64, 16, (9, 30), False, 1.0),      # bands of rows
    (37, 53, 40, (13,), True, 0.6),         # uneven last band
    (200, 24, 32, (5, 1, 1, 6), False, 1.0),   # bands of columns
    (19, 7, 128, (6, 2), True, 1.0),
    (33, 3, 512, (3,), False, 1.0),         # the most directions
    (150, 41, 24, (1030,), False, 1.0),     # more than one schedule upload
    (400, 130, 8, (8,), True, 1.0)])        # near the largest that fits
def test_equals_single_steps(nx, ny, q, parts, field, speed, walls, storage):
    args = (nx, ny, q, WALLS[walls], storage, parts)
    a = _run(*args, 0, field, speed, 11)
    b = _run(*args, 1, field, speed, 11)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
