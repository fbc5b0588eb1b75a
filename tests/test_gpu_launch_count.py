"""henry_launch_count: one per kernel launch, whatever the shape of its
blocks. The field statistics and the exceedance counts run blocks of 32 x G
threads (32 groups of samples on small grids, 8 on larger ones, fewer for a
few samples); a call is one launch each, a call of the QoI statistics too."""
import pytest

from paper_2403_17018_gb300 import binding as hb

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    hb.load()


@pytest.mark.parametrize("nx0,ny0,B", [(8, 4, 1), (8, 4, 64), (128, 64, 9)])
def test_a_statistics_call_counts_as_one_launch(nx0, ny0, B):
    ctx = hb.Context(hb.default_config(nx0=nx0, ny0=ny0, nlevels=1))
    n = nx0 * ny0
    c = torch.rand((B, n), dtype=torch.float64, device="cuda")
    q = torch.rand((B, hb.NQ), dtype=torch.float64, device="cuda")
    st = torch.zeros(B, dtype=torch.int32, device="cuda")
    acc = {k: v.reshape(n) for k, v in hb.new_field_accumulator(1, n).items()}
    count = torch.zeros(n, dtype=torch.int64, device="cuda")
    S = hb.LevelStats()
    for call in (lambda: ctx.field_stats(0, c, None, st, acc),
                 lambda: ctx.field_exceedance(0, c, st, 0.5, count),
                 lambda: ctx.level_stats(0, q, None, st, S)):
        before = ctx.launch_count()
        call()
        assert ctx.launch_count() - before == 1
