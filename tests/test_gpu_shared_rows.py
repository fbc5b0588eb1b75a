"""Tile heights that a schedule asks for (res_rows) on grids whose tiles warps
may share: heights of 16 and 64 rows are split between four warps for one
sample and for sixteen, 17 rows are not. The height changes the order of the sums that decide
convergence, not the equations; the batch changes nothing."""
import numpy as np
import pytest

from paper_2403_17018_gb300 import binding as hb

from gpu_helpers import xi_cuda
from test_gpu_parity import C_TOL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.load()


@pytest.mark.parametrize("precision", [hb.PREC_FP64, hb.PREC_FP32_MG])
def test_heights_and_batches_give_the_same_solutions(precision):
    xi = xi_cuda(0, 0, 16)
    ref = None
    for rows in (0, 16, 17, 64):
        cfg = hb.default_config(nx0=256, ny0=128, nlevels=1, nt0=2, T=450.0, precision=precision,
                                newton_rtol=1e-12, newton_atol=3e-13, newton_maxit=60,
                                newton_stag_tol=1e-11, jac_lag=30, res_rows=rows)
        got = []
        for B in (1, 16):
            out = hb.Context(cfg).solve(0, xi[:B].contiguous(), want_c=True, want_iters=True)
            assert out["status"].cpu().numpy().tolist() == [0] * B
            got.append({k: out[k][0].cpu().numpy() for k in ("c", "q", "iters")})
        assert all(np.array_equal(got[0][k], got[1][k]) for k in got[0]), rows
        ref = got[0]["c"] if ref is None else ref
        assert np.max(np.abs(got[0]["c"] - ref)) <= C_TOL
