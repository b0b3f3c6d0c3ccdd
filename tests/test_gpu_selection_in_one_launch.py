"""Fixed budget per head where the selection changes its form: the sizes at which a cluster gets more CTAs, a thread keeps
no more scores in registers, or three launches take over, and batches with one sequence far longer than the others.  Cut
values, lengths and rows exactly, against numpy (the check of test_gpu_select_and_recount)."""
import pytest

from paper_2601_07891_b200 import binding
from tests.test_gpu_select_and_recount import D, H, test_fixed_budget as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [
    [2047], [2048], [2049], [4096], [4097], [16384], [16385], [32768], [32769], [40960], [40961], [50000],
    [33000, 1, 0, 7], [81000, 900], [81000, 950], [20000] + [20] * 15, [30000] + [3] * 70])
@pytest.mark.parametrize("kind,ratio", [("normal", 0.25), ("low bits", 0.7), ("special", 1.0), ("same", 0.01)])
def test_cut_values(lens, kind, ratio):
    ctx = binding.Kvzap(256, 0, H, D, 1, max_tokens=sum(lens), max_seqs=len(lens))
    for window in (0, 128):
        check(ctx, lens, window, kind, ratio, False)
    ctx.close()


@pytest.mark.parametrize("lens,launches", [
    ([16000] + [20] * 2, 2), ([546] * 60, 2), ([200] * 200, 2), ([30000] + [20] * 20, 2), ([100000] + [20] * 9, 2),   # one
    ([50000] + [20] * 30, 4), ([100000] + [20] * 50, 4), ([120000] + [20] * 2, 2), ([300000] + [20] * 2, 4)])       # or three
def test_one_long_sequence_among_short_ones(lens, launches):
    """A few CTAs would count nearly all tokens of such a batch: three launches take it instead."""
    ctx = binding.Kvzap(256, 0, H, D, 1, max_tokens=sum(lens), max_seqs=len(lens))
    before = ctx.launch_count()
    check(ctx, lens, 128, "normal", 0.25, False)
    assert ctx.launch_count() - before == 2 * launches       # the check calls twice
    ctx.close()
