"""Start field: the stored float32 deviations are float32(float64(w_i) * dE) with
dE = e_eq(T_ref + dT) - e_eq(T_ref) in float64, over deviations from far below the split
product's range (where float64 decides) to hundreds of kelvin, and for cells without a
temperature.  The device's expm1 and the division may each be off by an ulp, which the
difference from e_ref leaves as an absolute error: |got - w dE| <= 2^-24 |w dE| + w 16 2^-53
(1 + e)^2 (e times its relative error, the exponent's error scaled by d ln e / d x = 1 + e)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
THETA, TREF = 624.8074248458514, 300.0


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("nx,ny,q", [(1, 1, 8), (33, 7, 24), (257, 65, 64), (40, 300, 1024)])
def test_start_field_is_the_rounded_product(nx, ny, q):
    import torch

    import paper_1911_00180_gb300 as wl
    rng = np.random.default_rng(nx + q)
    dT = (10.0 ** rng.uniform(-22, 2.4, (ny, nx)) * rng.choice([-1, 1], (ny, nx))).astype(np.float32)
    dT.flat[::7] = 0.0
    h = wl.WormLBM(nx, ny, q, mfp=8.0, bc=(0, 0, 0, 0), t_ref=TREF, theta=THETA)
    h.wlbm_init_temperature(torch.from_numpy(dT).cuda())
    got = h.wlbm_get_state().cpu().numpy()[:, 1:-1, 1:-1].astype(np.float64)
    w = wl.wlbm_lattice(q)[1].astype(np.float32).astype(np.float64)
    h.close()
    e = 1.0 / np.expm1(THETA / (TREF + dT.astype(np.float64)))
    de = e - 1.0 / np.expm1(THETA / TREF)
    want = w[:, None, None] * de
    tol = 2.0 ** -24 * np.abs(want) + w[:, None, None] * 16 * 2.0 ** -53 * (1 + e) ** 2
    assert np.all(np.abs(got - want) <= tol)
