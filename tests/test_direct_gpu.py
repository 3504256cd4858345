"""The direct-load step kernel against the TMA-tile kernel, which an explicit ring depth
selects: the same state bit for bit over the walls, storages and weight fields both take, at
sizes off the 32 x 8 cells of a block and with one cell in the last row or column of blocks;
and the direct-load reverse step (and recompute) against the variant-1 kernels, which sum in
another order: each of the steps' sums of Q terms may differ by Q roundings of 2^-24 of their
magnitude on either side, so gradients by n Q 2^-22 of the largest."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
P, I, A, S = W.PERIODIC, W.ISOTHERMAL, W.ADIABATIC_DIFFUSE, W.ADIABATIC_SPECULAR
CASES = [
    (289, 257, 32, (P, P, P, P), (0.0,) * 4, 1.0),
    (257, 130, 40, (I, S, A, A), (0.0, 0.0, 0.5, 0.0), 1.0),
    (160, 161, 64, (A, A, A, A), (0.0,) * 4, 0.6),
    (33, 300, 128, (I, I, P, P), (0.0,) * 4, 1.0),
    (31, 9, 512, (A, I, P, P), (0.3, 0.0, 0.0, 0.0), 1.0),
]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _grid(nx, ny, q, bc, spec, speed, storage, field):
    import paper_1911_00180_gb300 as wl
    kw = dict(mfp=6.0)
    if field:
        kw = dict(mfp_field=np.maximum(W.lognormal_mfp(nx, ny, seed=3, corr=4.0), 2.0))
    return wl.WormLBM(nx, ny, q, bc=bc, t_wall=(301.0, 300.0, 300.5, 300.0), specularity=spec,
                      speed=speed, storage=storage, **kw)


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("graph", [0, 6])
@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("nx,ny,q,bc,spec,speed", CASES)
def test_direct_step_equals_tma_step(nx, ny, q, bc, spec, speed, field, graph, storage):
    import torch

    from paper_1911_00180_gb300 import wlbm as api
    out = []
    for ring in (0, 8 if storage else (6 if q <= 64 else 4)):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            h = _grid(nx, ny, q, bc, spec, speed, storage, field)
            h.wlbm_set_option(api.OPT_RING_STAGES, ring)
            if ring and storage:
                h.wlbm_set_option(api.OPT_BF16_WIDE, 0)
            h.wlbm_set_option(api.OPT_GRAPH_STEPS, graph)
            h.wlbm_init_temperature(W.random_dT(nx, ny, seed=5, scale=0.5))
            h.wlbm_step(19)
            out.append([h.wlbm_get_state().cpu().numpy()[:, 1:-1, 1:-1]] +
                       [m.cpu().numpy() for m in h.wlbm_moments()])
            h.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("nx,ny,q,bc,spec,speed", CASES[:4] + [(700, 300, 32, (I, I, P, P), (0.0,) * 4, 1.0)])
def test_reverse_step_equals_variant_1(nx, ny, q, bc, spec, speed):
    import torch

    from paper_1911_00180_gb300 import wlbm as api
    n, out = 13, []
    gT = torch.from_numpy(np.random.default_rng(2).standard_normal((ny, nx)).astype(np.float32)).cuda()
    for variant in (3, 1):
        h = _grid(nx, ny, q, bc, spec, speed, 0, True)
        h.wlbm_set_option(api.OPT_STEP_VARIANT, variant)
        h.wlbm_adjoint_forward(W.random_dT(nx, ny, seed=5, scale=0.5), n, 5)
        g_mfp, g_tw, g_dT = h.wlbm_adjoint_backward(gT)
        out.append([g_mfp.cpu().numpy(), np.asarray(g_tw), g_dT.cpu().numpy()])
        h.close()
    for a, b in zip(*out):
        assert np.max(np.abs(a - b)) <= n * q * 2.0 ** -22 * max(np.max(np.abs(b)), 1e-30)
