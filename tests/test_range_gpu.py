"""The bfloat16 scale (max |e_eq(T) - e_ref| over the start field and the isothermal walls) from
the device's reduction of the start field, against numpy over every cell: odd sizes, a field at
an unaligned address, NaN cells (left out) and temperatures at or below 0 K (every cell
counts).  The scale is read from a checkpoint's header and must be the same float32."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
THETA, TREF = 624.8074248458514, 300.0
SCALE_AT = 8 + 6 * 4 + 4 * 4 + 4 * 4 + 4 * 8     # byte offset of the scale in the header


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1911_00180_gb300  # noqa: F401


def _delta(t):
    return 1.0 / np.expm1(THETA / t) - 1.0 / np.expm1(THETA / TREF)


@pytest.mark.parametrize("nx,ny,kind,shift", [
    (1, 1, "plain", 0), (3, 5, "plain", 1), (33, 31, "negative", 2), (1023, 7, "plain", 3),
    (640, 333, "nan", 0), (65, 17, "allnan", 1), (300, 41, "cold", 0)])
def test_scale(nx, ny, kind, shift):
    import torch
    import paper_1911_00180_gb300 as wl
    dT = W.random_dT(nx, ny, nx + ny, scale=3.0)
    if kind == "negative":
        dT = -np.abs(dT) - 1.0
    if kind == "nan":
        dT[::7, ::3] = np.nan
    if kind == "allnan":
        dT[:] = np.nan
    if kind == "cold":
        dT[5, 7] = -400.0
    buf = torch.zeros(nx * ny + 4, device="cuda")
    buf[shift:shift + nx * ny] = torch.from_numpy(dT.astype(np.float32).reshape(-1)).cuda()
    h = wl.WormLBM(nx, ny, 8, mfp=4.0, bc=(1, 1, 0, 0), t_wall=(300.5, 300.0, 300.0, 300.0),
                   storage=wl.STORE_BF16_DEV, theta=THETA)
    h.wlbm_init_temperature(buf[shift:shift + nx * ny].view(ny, nx))
    got = h.wlbm_save()[SCALE_AT:SCALE_AT + 4].view(np.float32)[0]
    h.close()
    v = dT.astype(np.float32).astype(np.float64)
    v = v[~np.isnan(v)]
    m = max([abs(_delta(300.5))] + ([np.abs(_delta(TREF + v)).max()] if v.size else []))
    assert abs(float(got) / float(np.float32(m)) - 1.0) <= 2.0 ** -23
