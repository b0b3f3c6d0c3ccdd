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
