"""Coarsest systems of every size that the direct solve takes: grids that are
their own coarsest level (4 to 64 unknowns, whole and partial warps of
columns, one and two elements per thread, 128 and 256 threads by the batch) and
grids above such a level, FP64 and FP32, against the FP64 oracle at the parity
tests' tolerance."""
import numpy as np
import pytest

from paper_2403_17018_gb300 import binding as hb

from gpu_helpers import oracle_solve, tight_config, xi_cuda
from test_gpu_parity import C_TOL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.load()


@pytest.mark.parametrize("precision", [hb.PREC_FP64, hb.PREC_FP32_MG])
@pytest.mark.parametrize("nx,ny", [(2, 2), (6, 2), (4, 3), (6, 3), (8, 3), (6, 5), (2, 16)])
@pytest.mark.parametrize("B", [3, 306])
def test_one_level_solves(nx, ny, B, precision):
    cfg = tight_config(nx0=nx, ny0=ny, nlevels=1, nt0=2, T=1800.0, precision=precision)
    ctx = hb.Context(cfg)
    assert ctx.level_info(0).n_mg == 1
    out = ctx.solve(0, xi_cuda(0, 0, B), want_c=True, want_iters=True)
    assert out["status"].cpu().numpy().tolist() == [0] * B
    for b in (0, B - 1):
        _, c_o, _ = oracle_solve(cfg, 0, xi_cuda(0, 0, B)[b].cpu().numpy())
        assert np.max(np.abs(out["c"][b].cpu().numpy() - c_o)) <= C_TOL


@pytest.mark.parametrize("precision", [hb.PREC_FP64, hb.PREC_FP32_MG])
@pytest.mark.parametrize("nx0,ny0", [(6, 3), (8, 3), (10, 3), (6, 5)])
def test_coarse_operators_beside_a_large_inverse(nx0, ny0, precision):
    cfg = tight_config(nx0=nx0, ny0=ny0, nlevels=3, nt0=1, T=1800.0, precision=precision)
    ctx = hb.Context(cfg)
    out = ctx.solve(2, xi_cuda(2, 0, 3), want_c=True)
    assert out["status"].cpu().numpy().tolist() == [0] * 3
    _, c_o, _ = oracle_solve(cfg, 2, xi_cuda(2, 0, 3)[1].cpu().numpy())
    assert np.max(np.abs(out["c"][1].cpu().numpy() - c_o)) <= C_TOL
