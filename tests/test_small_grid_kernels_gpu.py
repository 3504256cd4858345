"""Which kernel the default options of a small grid take, by the names the profiler records, and
the cluster launch where tests of equal bits had not reached it: more than 512 threads a block in
float32, several cells a thread, replayed graphs, and grids that change between cluster and
one-step launches; and the rule on steps and directions between the two.  The one-step launches (WLBM_OPT_TILE_LOOP) give the
same bits."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
P, I, A, S = W.PERIODIC, W.ISOTHERMAL, W.ADIABATIC_DIFFUSE, W.ADIABATIC_SPECULAR
WALLS = {"periodic": (P, P, P, P), "film": (I, I, A, A), "channel": (I, I, P, P),
         "square": (I, I, I, I), "duct": (P, P, A, I), "tube": (P, P, A, A)}


def _profile(run):
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        run()
        torch.cuda.synchronize()
    return [e.name for e in p.events() if "wlbm::" in e.name]


@pytest.fixture(scope="module")
def kernels():
    """kernels(run): names of the library's kernels that run() launches."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    h = _grid(16, 16, 8, WALLS["periodic"], 0)
    _profile(lambda: h.wlbm_step(1))            # the first session may record nothing
    h.close()

    def names(run):
        out = _profile(run)
        if not out:
            pytest.skip("the profiler records no kernels here")
        return out
    return names


def _grid(nx, ny, q, bc, storage, seed=3, spec=(0.0,) * 4, speed=1.0):
    import paper_1911_00180_gb300 as wl
    h = wl.WormLBM(nx, ny, q, mfp=6.0, bc=bc, t_wall=(301.0, 299.5, 300.5, 300.0), storage=storage,
                   specularity=spec, speed=speed)
    h.wlbm_init_temperature(W.random_dT(nx, ny, seed))
    return h


def _state(h, bc):
    y = slice(0 if bc[2] == A else 1, None if bc[3] == A else -1)
    return [h.wlbm_get_state().cpu().numpy()[:, y, 1:-1]] + [m.cpu().numpy() for m in
                                                             h.wlbm_moments()]


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,ny,q", [(2, 1, 8), (4, 2, 16), (64, 64, 16), (37, 53, 40), (200, 24, 32),
                                     (19, 7, 128), (33, 3, 512), (150, 41, 24)])
def test_cluster_launch_is_taken(kernels, nx, ny, q, storage):
    for bc in WALLS.values():
        h = _grid(nx, ny, q, bc, storage)
        before = h.wlbm_profile_read()[2]
        names = kernels(lambda: h.wlbm_step(7))
        assert len(names) == 1 and "k_step_cluster" in names[0], (bc, names)
        assert h.wlbm_profile_read()[2] == before + 1
        h.close()


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,ny,q,bc,spec,speed", [
    (289, 257, 32, (P, P, P, P), (0.0,) * 4, 1.0),
    (257, 130, 40, (I, S, A, A), (0.0, 0.0, 0.5, 0.0), 1.0),
    (160, 161, 64, (A, A, A, A), (0.0,) * 4, 0.6),
    (33, 300, 128, (I, I, P, P), (0.0,) * 4, 1.0),
    (31, 9, 512, (A, I, P, P), (0.3, 0.0, 0.0, 0.0), 1.0)])
def test_direct_kernels_are_taken(kernels, nx, ny, q, bc, spec, speed, storage):
    h = _grid(nx, ny, q, bc, storage, spec=spec, speed=speed)
    names = kernels(lambda: h.wlbm_step(3))
    assert sum("k_step_direct" in n for n in names) == 3, names
    if storage == 0:
        h.wlbm_adjoint_forward(W.random_dT(nx, ny, 5), 4, 2)
        names = kernels(lambda: h.wlbm_adjoint_backward(np.ones((ny, nx), np.float32)))
        assert sum("k_adj_direct" in n for n in names) == 4, names
    h.close()


@pytest.mark.parametrize("nx,ny,q,storage,walls,steps,kernel", [
    (128, 100, 8, 0, "periodic", 11, "k_step_cluster<float, 1024"),
    (128, 100, 8, 0, "film", 11, "k_step_cluster<float, 1024"),
    (130, 130, 16, 0, "duct", 33, "k_step_cluster<float, 1024"),       # two cells per thread
    (130, 130, 16, 0, "channel", 33, "k_step_cluster<float, 1024"),
    (128, 128, 32, 1, "film", 32, "k_step_cluster<__nv_bfloat16, 1024"),
    (1024, 16, 32, 1, "tube", 40, "k_step_cluster<__nv_bfloat16, 1024"),
    (130, 130, 16, 0, "periodic", 31, "k_step_direct<float"),          # too few steps
    (200, 100, 8, 0, "duct", 40, "k_step_direct<float"),               # too few directions
    (8176, 1, 8, 1, "tube", 40, "k_step_direct<__nv_bfloat16"),
    (40, 30, 24, 0, "film", 3, "k_step_direct<float"),
    (40, 30, 24, 0, "film", 4, "k_step_cluster<float"),
    (11, 11, 256, 0, "film", 1, "k_step_cluster<float"),
    (128, 16, 256, 1, "periodic", 1, "k_step_direct<__nv_bfloat16")])
def test_rule_and_equal_bits(kernels, nx, ny, q, storage, walls, steps, kernel):
    from paper_1911_00180_gb300 import wlbm as api
    bc, out = WALLS[walls], []
    for loop in (0, 1):
        h = _grid(nx, ny, q, bc, storage)
        h.wlbm_set_option(api.OPT_TILE_LOOP, loop)
        names = [k for k in kernels(lambda: h.wlbm_step(steps)) if "k_step" in k]
        assert loop or (len(names) == (1 if "cluster" in kernel else steps) and
                        all(kernel in k for k in names)), names
        h.wlbm_step(2)
        out.append(_state(h, bc))
        h.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("walls", ["periodic", "film"])
def test_graphs_and_changes_between_launches(kernels, walls, storage):
    import torch

    from paper_1911_00180_gb300 import wlbm as api
    bc, out = WALLS[walls], []
    for parts in (((12, 0, 41),), ((0, 0, 5), (0, 1, 3), (0, 0, 4), (12, 0, 12), (12, 1, 13), (0, 0, 4)),
                  ((0, 1, 41),)):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            h = _grid(60, 33, 24, bc, storage)
            for graph, loop, n in parts:
                h.wlbm_set_option(api.OPT_GRAPH_STEPS, graph)
                h.wlbm_set_option(api.OPT_TILE_LOOP, loop)
                r0 = h.wlbm_get_option(api.OPT_GRAPH_REPLAYS)
                names = kernels(lambda: h.wlbm_step(n)) if graph == 0 else h.wlbm_step(n) or []
                assert all(("k_step_cluster" in k) == (loop == 0 and n >= 4)
                           for k in names if "k_step" in k), names
                assert h.wlbm_get_option(api.OPT_GRAPH_REPLAYS) - r0 == (n // 12 if graph else 0)
            out.append(_state(h, bc))
            h.close()
    for k in (0, 1):
        for a, b in zip(out[k], out[2]):
            assert np.array_equal(a, b)
