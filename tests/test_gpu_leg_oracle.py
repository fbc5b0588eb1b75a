"""V-cycles of one launch per leg (k_leg) against the FP64 oracle, on a single
strip of 32 lanes in several chunks of rows (64x32 cells x 300) and on strips
that end inside the grid (192x160 cells x 75), both on settings where the
cycles converge. With no fused kernel on any level the launch count says
whether the legs were taken: they are the only difference between mg_fusion
= 1 and 0 here, and replace four or five launches each.

V-cycles without pre-sweeps (nu1 = 0) restrict the residuals of all four
children of a coarse cell from an iterate that has seen no red half-sweep: the
launches per operation against the fused kernel on 32x16 cells, which computes
the same cycle bit for bit, and both against the oracle."""
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


def _both(level, B, **kw):
    """The solve with mg_fusion 0 and 1: outputs and launches of each."""
    res, launches = [], []
    for fusion in (0, 1):
        cfg = tight_config(mg_fusion=fusion, **kw)
        ctx = hb.Context(cfg)
        res.append(ctx.solve(level, xi_cuda(level, 0, B), want_c=True, want_p=True, want_iters=True))
        torch.cuda.synchronize()
        launches.append(ctx.launch_count())
    for out in res:
        assert out["status"].cpu().numpy().tolist() == [0] * B
        assert all(bool(torch.isfinite(out[k]).all()) for k in ("c", "p", "q"))
    for k in ("c", "p", "q", "iters"):
        assert torch.equal(res[0][k], res[1][k]), k
    return cfg, res[1], launches


@pytest.mark.parametrize("nx,ny,B,nt,T", [(64, 32, 300, 2, 1800.0), (192, 160, 75, 1, 56.25)])
def test_legs_match_the_oracle(nx, ny, B, nt, T):
    cfg, out, launches = _both(0, B, nx0=nx, ny0=ny, nlevels=1, nt0=nt, T=T, vcycles=2,
                               precision=hb.PREC_FP32_MG, mg_small_cells=0, mg_cluster_cells=0,
                               mg_tb_cells=0)
    assert launches[1] < launches[0]
    for b in (0, B - 1):
        _, c_o, _ = oracle_solve(cfg, 0, xi_cuda(0, 0, B)[b].cpu().numpy())
        assert np.max(np.abs(out["c"][b].cpu().numpy() - c_o)) <= C_TOL


@pytest.mark.parametrize("precision", [hb.PREC_FP64, hb.PREC_FP32_MG])
@pytest.mark.parametrize("level,cycles,kry", [(0, 3, 0), (0, 1, 4), (1, 3, 0)])
def test_cycles_without_pre_sweeps(precision, level, cycles, kry):
    cfg, out, launches = _both(level, 3, nlevels=2, nt0=1, T=1800.0, precision=precision, nu1=0,
                               nu2=2, vcycles=cycles, krylov_iters=kry, mg_small_cells=512,
                               mg_tb_cells=0)
    assert launches[1] < launches[0]
    for b in (0, 2):
        _, c_o, _ = oracle_solve(cfg, level, xi_cuda(level, 0, 3)[b].cpu().numpy())
        assert np.max(np.abs(out["c"][b].cpu().numpy() - c_o)) <= C_TOL
