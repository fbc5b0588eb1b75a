"""Batch statistics at the edges of their sample groups: batches of 1 to 70
samples (fewer than, equal to and not a multiple of the groups), leading
samples that failed, grids that do not fill a block of 32 cells, a running
state that is continued. Against two-pass numpy in FP64; the counts exactly.
Tolerance 1e-12 of the largest value: rounding of sums of at most 100 terms."""
import numpy as np
import pytest

from paper_2403_17018_gb300 import binding as hb

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.load()


@pytest.mark.parametrize("nx0,ny0,level", [(12, 6, 0), (6, 3, 1), (32, 16, 1)])
@pytest.mark.parametrize("B,bad", [(1, 0), (2, 1), (9, 8), (33, 12), (70, 0)])
def test_batches_match_two_pass_numpy(nx0, ny0, level, B, bad):
    ctx = hb.Context(hb.default_config(nx0=nx0, ny0=ny0, nlevels=2))
    li = ctx.level_info(level)
    n = li.nx * li.ny
    rng = np.random.default_rng(B * 100 + nx0)
    c = 0.7 + 1e-3 * rng.standard_normal((2, B, n))
    cc = 0.7 + 1e-3 * rng.standard_normal((2, B, n // 4)) if level else None
    q = 300.0 + rng.standard_normal((2, B, hb.NQ))
    qc = q + 1e-2 * rng.standard_normal(q.shape) if level else None
    st = np.zeros(B, dtype=np.int32)
    st[:bad] = 1
    acc = {k: v.reshape(n) for k, v in hb.new_field_accumulator(1, n).items()}
    count = torch.zeros(n, dtype=torch.int64, device="cuda")
    S = hb.LevelStats()
    cu = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
    for k in range(2):
        ctx.level_stats(level, cu(q[k]), cu(qc[k]) if level else None, cu(st), S)
        ctx.field_stats(level, cu(c[k]), cu(cc[k]) if level else None, cu(st), acc)
        ctx.field_exceedance(level, cu(c[k]), cu(st), 0.7, count)
    ok = st == 0
    m = 2 * int(ok.sum())
    f = c[:, ok].reshape(m, n)
    d = f
    if level:
        up = cc.reshape(2, B, li.ny // 2, li.nx // 2).repeat(2, axis=2).repeat(2, axis=3)
        d = (c - up.reshape(2, B, n))[:, ok].reshape(m, n)
    assert np.array_equal(acc["n"].cpu().numpy(), np.full(n, m))
    assert np.array_equal(count.cpu().numpy(), (f > 0.7).sum(axis=0))
    s = S.numpy()
    assert s["n"] == m
    if m == 0:
        return
    qf = q[:, ok].reshape(m, -1)
    qd = (q - qc)[:, ok].reshape(m, -1) if level else qf
    den = max(m - 1, 1)
    for got, x in ((acc["mean_f"], f.mean(0)), (acc["m2_f"], ((f - f.mean(0)) ** 2).sum(0)),
                   (acc["mean_d"], d.mean(0)), (acc["m2_d"], ((d - d.mean(0)) ** 2).sum(0)),
                   (s["mean_f"], qf.mean(0)), (s["var_f"], ((qf - qf.mean(0)) ** 2).sum(0) / den),
                   (s["mean_d"], qd.mean(0)), (s["var_d"], ((qd - qd.mean(0)) ** 2).sum(0) / den)):
        got = got.cpu().numpy() if hasattr(got, "cpu") else got
        assert np.max(np.abs(got - x)) <= 1e-12 * max(np.max(np.abs(x)), 1e-12)


def test_exceedance_orders_doubles():
    """Zeros of both signs, infinities, denormals and NaN compare as doubles."""
    ctx = hb.Context(hb.default_config(nx0=8, ny0=4, nlevels=1))
    v = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -np.nan, 5e-324, -5e-324] * 4)
    c = torch.from_numpy(v[None].copy()).cuda()
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    for th in (0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, 5e-324):
        count = torch.zeros(32, dtype=torch.int64, device="cuda")
        ctx.field_exceedance(0, c, st, th, count)
        with np.errstate(invalid="ignore"):
            assert np.array_equal(count.cpu().numpy(), (v > th).astype(np.int64)), th
