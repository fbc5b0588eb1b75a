"""henry_debug_copy's face fluxes (11 qx, 12 qy) after a solve: on the finest
level those of the last residual, hence of the solution, with and without
operator reuse and also where the V-cycles run in one launch per leg; on the
coarser levels the sums of the next finer level's at the last rebuild of the
operators.

Tolerance: a flux is t (p_U - p_L + rho terms) with the operands taken from the
solver's own arrays, a handful of roundings of terms no larger than max t
times the largest difference of p or of the hydrostatic term: 8 ulp of that."""
import numpy as np
import pytest

from paper_2403_17018_gb300 import binding as hb

from gpu_helpers import xi_cuda

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.load()


# (nx, ny, samples): 64x32 x 2 (launches per operation and the fused kernel), 64x32 x 300
# and 1024x512 x 16 (legs, on the latter's two finest levels), 6x5 (one level)
@pytest.mark.parametrize("nx,ny,B", [(64, 32, 2), (64, 32, 300), (1024, 512, 16), (6, 5, 3)])
@pytest.mark.parametrize("jac_lag", [0, 30])
@pytest.mark.parametrize("precision", [hb.PREC_FP64, hb.PREC_FP32_MG])
def test_fluxes_belong_to_the_solution(nx, ny, B, jac_lag, precision):
    if nx == 1024 and precision == hb.PREC_FP64:
        pytest.skip("the legs are FP32")
    cfg = hb.default_config(nx0=nx, ny0=ny, nlevels=1, nt0=1, T=56.25, precision=precision,
                            jac_lag=jac_lag, mg_small_cells=32, mg_cluster_cells=0, mg_tb_cells=0)
    ctx = hb.Context(cfg)
    top = ctx.level_info(0).n_mg - 1
    out = ctx.solve(0, xi_cuda(0, 0, B), want_c=True, want_p=True)
    assert out["status"].cpu().numpy().tolist() == [0] * B

    def get(k, what):
        w, h = nx >> (top - k), ny >> (top - k)
        a = ctx.debug_copy(0, 0, k, what, B * w * h * 8).view(np.float64)
        return a.reshape(B, h, w)

    p, c, tx, ty, qx, qy = (get(top, w) for w in (3, 4, 7, 9, 11, 12))
    assert np.array_equal(c, out["c"].cpu().numpy())
    dr, hy = cfg.rho1 - cfg.rho0, cfg.Ly / ny
    y = (np.arange(ny) + 0.5) * hy
    p_right = (dr * cfg.g * (cfg.Ly - y))[None, :, None]          # reduced seawater pressure
    dp = np.diff(np.concatenate([p, np.broadcast_to(p_right, (B, ny, 1))], axis=2), axis=2)
    tol = 8 * np.finfo(float).eps
    assert np.max(np.abs(qx + tx * dp)) <= tol * np.max(tx) * np.max(np.abs(p))
    if ny > 1:
        buoy = 0.5 * dr * (c[:, :-1] + c[:, 1:]) * cfg.g * hy
        want = -ty[:, :-1] * (np.diff(p, axis=1) + buoy)
        assert np.max(np.abs(qy[:, :-1] - want)) <= tol * np.max(ty[:, :-1]) * np.max(np.abs(p))
    assert np.all(qy[:, -1] == 0.0)
    for k in range(top - 1, 0, -1):
        fx, fy = get(k, 11), get(k, 12)
        assert np.array_equal(get(k - 1, 11), fx[:, 0::2, 1::2] + fx[:, 1::2, 1::2])
        assert np.array_equal(get(k - 1, 12), fy[:, 1::2, 0::2] + fy[:, 1::2, 1::2])
