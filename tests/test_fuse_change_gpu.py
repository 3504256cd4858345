"""WLBM_OPT_FUSE_PERIODIC may be set at any step, and on a handle that loads a checkpoint: steps
whose kernel mirrors the edges start from copies of the present state, whatever ran before."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
NX, NY, Q = 45, 38, 24


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _handle(storage, fuse):
    import paper_1911_00180_gb300 as wl
    h = wl.WormLBM(NX, NY, Q, mfp=6.0, bc=(0,) * 4, t_wall=(300.0,) * 4, storage=storage)
    h.wlbm_set_option(wl.wlbm.OPT_STEP_VARIANT, 1)
    h.wlbm_set_option(wl.wlbm.OPT_FUSE_PERIODIC, fuse)
    h.wlbm_init_temperature(W.random_dT(NX, NY, 4))
    return h


def _bits(h):
    return h.wlbm_get_state().cpu().numpy()[:, 1:-1, 1:-1]


@pytest.mark.parametrize("storage", [0, 1])
def test_single_grid(storage):
    from paper_1911_00180_gb300 import wlbm as api
    h = _handle(storage, 0)
    h.wlbm_step(17)
    want = _bits(h)
    h.close()
    h = _handle(storage, 0)
    for fuse, n in ((0, 5), (1, 4), (0, 3)):
        h.wlbm_set_option(api.OPT_FUSE_PERIODIC, fuse)
        h.wlbm_step(n)
    blob = h.wlbm_save()
    h.close()
    h = _handle(storage, 1)
    h.wlbm_step(2)
    h.wlbm_load(blob)
    h.wlbm_step(5)
    assert np.array_equal(_bits(h), want)
    h.close()


@pytest.mark.parametrize("storage", [0, 1])
def test_batch(storage):
    import paper_1911_00180_gb300 as wl
    from paper_1911_00180_gb300 import wlbm as api
    specs = [dict(nx=NX + 7 * k, ny=NY, q=Q, mfp=6.0, bc=(0,) * 4, t_wall=(300.0,) * 4)
             for k in range(3)]
    out = []
    for parts in (((0, 17),), ((0, 5), (1, 4), (0, 3), (1, 5))):
        b = wl.WormLBMBatch(specs, storage=storage)
        b.wlbm_batch_set_option(api.OPT_STEP_VARIANT, 1)
        b.wlbm_batch_init_temperature([W.random_dT(p["nx"], p["ny"], 4) for p in specs])
        for fuse, n in parts:
            b.wlbm_batch_set_option(api.OPT_FUSE_PERIODIC, fuse)
            b.wlbm_batch_step(n)
        out.append([_bits(v) for v in b.instances])
        b.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
