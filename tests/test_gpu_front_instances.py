"""Every instance of the per-sequence kernel for split sequences (2, 4, 8 and 16 blocks to a sequence, 4, 8 and 16 tokens to a thread, as
148 SMs choose them), with sequences far shorter than the longest and empty ones among them, and batches that take one kernel per step:
sequences beyond the largest, and one more of those that need 16 blocks than run at once. Decided in fp32 with one rounding per operation on both sides: every index is the oracle's."""
import pytest

from test_gpu_front_slices import PATS, _check
from test_gpu_steps import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fast", [True, False])
@pytest.mark.parametrize("lengths", [
    [20000] * 36 + [0, 1, 700, 19999],                                                            # 2 blocks, 16 tokens a thread
    [16000] * 17 + [15999, 0, 33], [20000] * 17 + [130, 1, 19999], [40000] * 16 + [0, 39999],      # 4 blocks: 4, 8, 16
    [20000] * 6 + [2049, 1], [40000] * 7 + [0, 65], [70000] * 6 + [5, 69999],                     # 8 blocks: 4, 8, 16
    [33000, 16, 0], [70000, 1, 40], [140000, 3000],                                               # 16 blocks: 4, 8, 16
    [262145, 20, 5000], [140000] * 7 + [131073]], ids=lambda v: f"{len(v)}x{max(v)}")
def test_instances(lengths, fast):
    _check(_workload(lengths, PATS, spans=[6, 64, 33, 12], seed=len(lengths), Hq=1, Hkv=1, W=32), 48, fast)
