"""Batches whose samples agree: cells counted below a threshold, boxes that no
salt reaches, levels whose difference is the same for every sample. Their mean
is the value and their variance zero, exactly, and no batch has a negative
variance (its square root goes into the sample allocation). The values of the
first three are ones whose rounded sum over the batch is not a multiple of
the value, so that deviations from the mean of sums do not vanish."""
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


@pytest.mark.parametrize("B,value", [(459, 6.6068620696728679), (884, 7.6512982843585888),
                                     (890, 7.287119020758567), (1, 0.1), (7, 1.0 / 3.0), (300, 0.0)])
@pytest.mark.parametrize("level,bad", [(0, 0), (1, 0), (1, 5)])
def test_constant_batches_have_no_variance(B, value, level, bad):
    ctx = hb.Context(hb.default_config(nx0=8, ny0=4, nlevels=2))
    li = ctx.level_info(level)
    n = li.nx * li.ny
    st = torch.zeros(B + bad, dtype=torch.int32, device="cuda")
    st[:bad] = 2
    full = lambda v, *shape: torch.full((B + bad,) + shape, v, dtype=torch.float64, device="cuda")
    q, c = full(value, hb.NQ), full(value, n)
    qc = full(0.75 * value, hb.NQ) if level else None
    cc = full(0.75 * value, n // 4) if level else None
    for t in (q, c) + ((qc, cc) if level else ()):
        t[:bad] = float("nan")
    acc = {k: v.reshape(n) for k, v in hb.new_field_accumulator(1, n).items()}
    S = hb.LevelStats()
    for _ in range(2):                       # the second batch is merged into the first
        ctx.level_stats(level, q, qc, st, S)
        ctx.field_stats(level, c, cc, st, acc)
    d = value - 0.75 * value if level else value
    s = S.numpy()
    assert s["n"] == 2 * B
    for mean, var, v in ((s["mean_f"], s["var_f"], value), (s["mean_d"], s["var_d"], d),
                         (acc["mean_f"].cpu().numpy(), acc["m2_f"].cpu().numpy(), value),
                         (acc["mean_d"].cpu().numpy(), acc["m2_d"].cpu().numpy(), d)):
        assert np.all(mean == v) and np.all(var == 0.0)


@pytest.mark.parametrize("B", [3, 257, 600])
def test_last_bit_noise_has_no_negative_variance(B):
    ctx = hb.Context(hb.default_config(nx0=8, ny0=4, nlevels=1))
    rng = np.random.default_rng(B)
    v = rng.uniform(0.1, 10.0, 32)
    x = np.where(rng.random((B, 32)) < 0.5, v, np.nextafter(v, 100.0))
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    S = ctx.level_stats(0, torch.from_numpy(x[:, :hb.NQ].copy()).cuda(), None, st, hb.LevelStats())
    acc = {k: t.reshape(32) for k, t in hb.new_field_accumulator(1, 32).items()}
    ctx.field_stats(0, torch.from_numpy(x).cuda(), None, st, acc)
    assert np.all(S.numpy()["var_f"] >= 0.0) and np.all(acc["m2_f"].cpu().numpy() >= 0.0)
