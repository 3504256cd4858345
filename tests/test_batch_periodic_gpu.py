"""The batched periodic pass' block table: written once, so that WLBM_OPT_FUSE_PERIODIC touches no
device (it can be set while the batch's stream is being captured), and instances that a fused
step kernel mirrors itself may stand anywhere in the batch."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
P, I, A = W.PERIODIC, W.ISOTHERMAL, W.ADIABATIC_DIFFUSE
T = (301.0, 300.0, 300.5, 300.0)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _specs():
    return [dict(nx=nx, ny=ny, q=q, mfp=6.0, bc=bc, t_wall=T) for nx, ny, q, bc in (
        (65, 40, 32, (P, P, P, P)), (30, 50, 64, (I, I, P, P)), (1, 9, 8, (P, P, P, P)),
        (300, 7, 16, (P, P, A, A)), (40, 20, 24, (I, I, A, A)), (129, 33, 40, (P, P, P, P)))]


def _run(options, steps):
    import torch

    import paper_1911_00180_gb300 as wl
    specs = _specs()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        b = wl.WormLBMBatch(specs, stream=s)
        for key, value in options:
            b.wlbm_batch_set_option(key, value)
        b.wlbm_batch_init_temperature([W.random_dT(p["nx"], p["ny"], 7 + k)
                                       for k, p in enumerate(specs)])
        b.wlbm_batch_step(steps)
        out = [v.wlbm_get_state().cpu().numpy()[:, 1:-1, 1:-1] for v in b.instances]
        b.close()
    return out


def test_fused_or_not_gives_the_same_states():
    from paper_1911_00180_gb300 import wlbm as api
    v1, fuse = (api.OPT_STEP_VARIANT, 1), (api.OPT_FUSE_PERIODIC, 1)
    plain = _run([v1], 15)
    for options in ([v1, fuse], [fuse, v1], [fuse, v1, (api.OPT_FUSE_PERIODIC, 0)]):
        for a, b in zip(plain, _run(options, 15)):
            assert np.array_equal(a, b)


def test_fuse_option_during_capture():
    import torch

    import paper_1911_00180_gb300 as wl
    from paper_1911_00180_gb300 import wlbm as api
    s = torch.cuda.Stream()
    x = torch.ones(64, device="cuda")
    with torch.cuda.stream(s):
        b = wl.WormLBMBatch(_specs(), stream=s)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            x.add_(1.0)
            b.wlbm_batch_set_option(api.OPT_FUSE_PERIODIC, 1)
            x.add_(1.0)
        g.replay()
        s.synchronize()
        assert b.wlbm_batch_get_option(api.OPT_FUSE_PERIODIC) == 1
        assert float(x[0]) == 3.0
        b.close()
