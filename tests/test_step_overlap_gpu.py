"""Kernels of consecutive steps overlap (programmatic dependent launches): n steps in one call
must equal, bit for bit, n calls of one step with a device synchronisation after each, for
grids on both sides of the sizes at which the kernels of a step change, with graphs and in
batches (all-periodic ones and mixed ones)."""
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


def _steps(h, n, one, step):
    import torch
    if not one:
        step(n)
    else:
        for _ in range(n):
            step(1)
            torch.cuda.synchronize()


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,ny,q,bc", [
    (300, 400, 24, (P, P, P, P)), (1100, 500, 16, (P, P, P, P)), (2049, 1030, 8, (P, P, P, P)),
    (700, 600, 16, (I, I, A, A)), (515, 260, 32, (A, A, A, A)), (900, 700, 8, (I, I, P, P))])
def test_steps_equal_synchronised_steps(nx, ny, q, bc, storage):
    import torch

    import paper_1911_00180_gb300 as wl
    from paper_1911_00180_gb300 import wlbm as api
    out = []
    for one, graph in ((True, 0), (False, 0), (False, 6)):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            h = wl.WormLBM(nx, ny, q, mfp=5.0, bc=bc, t_wall=(301.0, 300.0, 300.0, 300.0),
                           storage=storage)
            h.wlbm_set_option(api.OPT_GRAPH_STEPS, graph)
            h.wlbm_init_temperature(W.random_dT(nx, ny, seed=4, scale=0.5))
            _steps(h, 25, one, h.wlbm_step)
            out.append(h.wlbm_get_state().cpu().numpy()[:, 1:-1, 1:-1])
            h.close()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("walls", ["periodic", "mixed"])
def test_batch_steps_equal_synchronised_steps(walls, storage):
    import torch

    import paper_1911_00180_gb300 as wl
    from paper_1911_00180_gb300 import wlbm as api
    per, film = (P, P, P, P), (I, I, A, A)
    sizes = [(257, 33, 32, per, 4.0), (31, 130, 8, per, 9.0)]
    sizes += [(1500, 1450, 8, per, 9.0), (129, 15, 64, per, 9.0)] if walls == "periodic" else [
        (129, 15, 64, (I, I, P, P), 9.0), (140, 41, 16, film, 3.0)]
    specs = [dict(nx=nx, ny=ny, q=q, bc=bc, mfp=mfp, t_wall=(301.0, 300.0, 300.0, 300.0))
             for nx, ny, q, bc, mfp in sizes]
    out = []
    for one, graph in ((True, 0), (False, 0), (False, 6)):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            b = wl.WormLBMBatch(specs, storage=storage, stream=s)
            b.wlbm_batch_set_option(api.OPT_GRAPH_STEPS, graph)
            b.wlbm_batch_init_temperature([W.random_dT(c["nx"], c["ny"], seed=k, scale=0.5)
                                           for k, c in enumerate(specs)])
            _steps(b, 25, one, b.wlbm_batch_step)
            out.append([v.wlbm_get_state().cpu().numpy()[:, 1:-1, 1:-1] for v in b.instances])
            b.close()
    for got in out[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(out[0], got))
