"""k_residual at the edges of its tiles: one, two and four columns per thread,
grids narrower and wider than a warp's columns (64 and 128), rows that do not
fill a tile, pointers that rule out vector loads. Against the FP64 oracle,
with the tolerances of the parity tests (1e-12 of the flux scale for R, 1e-11
of a block's largest entry for J: rounding of a few dozen FP64 operations)."""
import numpy as np
import pytest

from oracle import henry as H
from paper_2403_17018_gb300 import binding as hb
from paper_2403_17018_gb300.inputs import xi_batch

from gpu_helpers import oracle_physics
from test_gpu_parity import _oracle_jacobian_blocks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.load()


def _states(nx, ny, B):
    cfg = hb.default_config()
    ph = oracle_physics(cfg)
    g = H.Grid(nx=nx, ny=ny, nt=1, T=1800.0)
    rng = np.random.default_rng(100 * nx + ny)
    out = {k: [] for k in ("phi", "K", "qin", "p", "c", "c_old")}
    for b in range(B):
        f = H.fields(g, ph, xi_batch(0, 7, B)[b])
        c = np.clip(rng.random((ny, nx)), 0, 1)
        for k, v in (("phi", f.phi), ("K", f.K), ("qin", f.qin), ("c", c),
                     ("c_old", np.clip(c + 0.1 * rng.standard_normal((ny, nx)), 0, 1)),
                     ("p", H.hydrostatic_guess(g, ph) + 40 * rng.standard_normal((ny, nx)))):
            out[k].append(v)
    return cfg, ph, g, {k: np.array(v) for k, v in out.items()}


def _cuda_tensor(a, offset=0):
    """a on the GPU, its data `offset` doubles off an allocation's start."""
    buf = torch.empty(a.size + offset, dtype=torch.float64, device="cuda")
    t = buf[offset:].view(a.shape)
    t.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return t


@pytest.mark.parametrize("nx,ny", [(2, 1), (3, 5), (62, 9), (64, 8), (66, 3), (130, 17), (131, 4)])
def test_residual_tiles_match_the_oracle(nx, ny):
    cfg, ph, g, s = _states(nx, ny, 2)
    t = {k: _cuda_tensor(v) for k, v in s.items()}
    R, J = hb.residual_jacobian(cfg, g.tau, *(t[k] for k in ("phi", "K", "qin", "p", "c", "c_old")))
    R0, none = hb.residual_jacobian(cfg, g.tau, *(t[k] for k in ("phi", "K", "qin", "p", "c", "c_old")),
                                    want_J=False)
    assert none is None and (R0 - R).abs().max() <= 1e-14 * R.abs().max()
    R, J = R.cpu().numpy(), J.cpu().numpy()
    for b in range(2):
        f = H.Fields(phi=s["phi"][b], K=s["K"][b], qin=s["qin"][b])
        st = (s["p"][b], s["c"][b], s["c_old"][b])
        want = H.residual(g, ph, f, *st)
        fx = H.face_fluxes(g, ph, f, s["p"][b], s["c"][b])
        scale = max([np.max(np.abs(v)) for v in (fx["mass_x"], fx["mass_y"], want[0]) if v.size])
        for e in range(2):
            assert np.max(np.abs(R[b, e] - want[e])) <= 1e-12 * scale
        Jo = _oracle_jacobian_blocks(H.jacobian(g, ph, f, *st), nx, ny)
        for m in range(20):
            assert np.max(np.abs(J[b, m] - Jo[m])) <= 1e-11 * max(np.max(np.abs(Jo[m])), 1e-300), (b, m)


def test_unaligned_pointers_take_the_scalar_path():
    """The same states 8 bytes off a 16-byte boundary: no vector loads, the
    same equations (the roundings of the two forms differ)."""
    cfg, _, g, s = _states(66, 5, 2)
    names = ("phi", "K", "qin", "p", "c", "c_old")
    a = hb.residual_jacobian(cfg, g.tau, *(_cuda_tensor(s[k]) for k in names))
    b = hb.residual_jacobian(cfg, g.tau, *(_cuda_tensor(s[k], 1) for k in names))
    for x, y in zip(a, b):
        assert (x - y).abs().max() <= 1e-13 * x.abs().max()
