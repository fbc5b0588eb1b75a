"""k_residual on widths that fill a warp with several row groups (8, 10, 6 or 16
lanes per row, two or four columns per lane), and tall tiles shared by four,
two or one warps by the batch.

Residual and Jacobian in the natural layout against the FP64 oracle with the
tolerances of the parity tests; solves (residual-only form, operators reused)
against the oracle's; and the tall tiles' sums, which decide convergence, by
the bits of a sample's solution and its iteration count in batches of 1, 8
and 16 (four, two and one warps per tile)."""
import numpy as np
import pytest

from oracle import henry as H
from paper_2403_17018_gb300 import binding as hb

from gpu_helpers import oracle_solve, tight_config, xi_cuda
from test_gpu_parity import C_TOL, _oracle_jacobian_blocks
from test_gpu_residual_tiles import _cuda_tensor, _states

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.load()


@pytest.mark.parametrize("nx,ny", [(80, 7), (48, 10), (36, 24), (112, 5), (134, 6), (45, 9)])
def test_row_groups_match_the_oracle(nx, ny):
    cfg, ph, g, s = _states(nx, ny, 2)
    t = [_cuda_tensor(s[k]) for k in ("phi", "K", "qin", "p", "c", "c_old")]
    R, J = (a.cpu().numpy() for a in hb.residual_jacobian(cfg, g.tau, *t))
    for b in range(2):
        f = H.Fields(phi=s["phi"][b], K=s["K"][b], qin=s["qin"][b])
        st = (s["p"][b], s["c"][b], s["c_old"][b])
        want = H.residual(g, ph, f, *st)
        fx = H.face_fluxes(g, ph, f, s["p"][b], s["c"][b])
        scale = max(np.max(np.abs(v)) for v in (fx["mass_x"], fx["mass_y"], want[0]))
        for e in range(2):
            assert np.max(np.abs(R[b, e] - want[e])) <= 1e-12 * scale
        Jo = _oracle_jacobian_blocks(H.jacobian(g, ph, f, *st), nx, ny)
        for m in range(20):
            assert np.max(np.abs(J[b, m] - Jo[m])) <= 1e-11 * max(np.max(np.abs(Jo[m])), 1e-300), (b, m)


@pytest.mark.parametrize("precision", [hb.PREC_FP64, hb.PREC_FP32_MG])
@pytest.mark.parametrize("nx,ny,jac_lag,res_rows", [(80, 24, 10, 0), (80, 24, 0, 0), (160, 48, 10, 0),
                                                    (160, 48, 10, 5), (96, 48, 0, 3)])
def test_solves_match_the_oracle(nx, ny, jac_lag, res_rows, precision):
    cfg = tight_config(nx0=nx, ny0=ny, nlevels=1, nt0=2, T=900.0, precision=precision,
                       jac_lag=jac_lag, res_rows=res_rows)
    out = hb.Context(cfg).solve(0, xi_cuda(0, 0, 3), want_c=True)
    assert out["status"].cpu().numpy().tolist() == [0] * 3
    _, c_o, _ = oracle_solve(cfg, 0, xi_cuda(0, 0, 3)[2].cpu().numpy())
    assert np.max(np.abs(out["c"][2].cpu().numpy() - c_o)) <= C_TOL


@pytest.mark.parametrize("precision", [hb.PREC_FP64, hb.PREC_FP32_MG])
def test_shared_tiles_do_not_depend_on_the_batch(precision):
    xi = xi_cuda(0, 0, 16)
    cfg = hb.default_config(nx0=512, ny0=256, nlevels=1, nt0=2, T=225.0, precision=precision, jac_lag=30)
    first = None
    for B in (1, 8, 16):
        out = hb.Context(cfg).solve(0, xi[:B].contiguous(), want_c=True, want_p=True, want_iters=True)
        assert out["status"].cpu().numpy().tolist() == [0] * B
        got = {k: out[k][0].cpu().numpy() for k in ("c", "p", "q", "iters")}
        first = first or got
        assert all(np.array_equal(got[k], first[k]) for k in got), B
