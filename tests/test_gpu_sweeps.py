"""The launches per operation of a V-cycle (k_smooth, k_resid_restrict,
k_prolong, k_update: a grid row per sample, positions split into row and
column by a multiplication, the first red half-sweep replaced by the guess's
writer) on grids whose widths are no powers of two, with and without pre- and
post-sweeps, against the FP64 oracle at the parity tests' tolerance."""
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
@pytest.mark.parametrize("nx0,ny0,level,nu,cycles", [(10, 3, 3, (2, 2), 2), (14, 2, 3, (1, 2), 2),
                                                     (6, 5, 3, (0, 2), 3), (6, 5, 2, (2, 0), 3)])
def test_launches_per_operation_match_the_oracle(precision, nx0, ny0, level, nu, cycles):
    cfg = tight_config(nx0=nx0, ny0=ny0, nlevels=level + 1, nt0=1, T=1800.0, mg_fusion=0,
                       precision=precision, nu1=nu[0], nu2=nu[1], vcycles=cycles)
    ctx = hb.Context(cfg)
    xi = xi_cuda(level, 0, 3)
    out = ctx.solve(level, xi, want_c=True)
    if nu == (0, 2):   # no pre-sweeps: the cycles diverge on these grids, and say so
        assert out["status"].cpu().numpy().tolist() == [2, 2, 2]
        return
    assert out["status"].cpu().numpy().tolist() == [0, 0, 0]
    for b in (0, 2):
        _, c_o, _ = oracle_solve(cfg, level, xi[b].cpu().numpy())
        assert np.max(np.abs(out["c"][b].cpu().numpy() - c_o)) <= C_TOL
