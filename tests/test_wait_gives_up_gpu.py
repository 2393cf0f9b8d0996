"""A wait that gives up because something else has failed: its CTA hears of it as of one that runs out."""
import pytest

from paper_2505_19602_b200 import binding

pytestmark = pytest.mark.gpu


def test_a_wait_on_a_failed_context_tells_its_cta():
    sides = (1, 2)
    kv = binding.ScaleKV(1, 1, 1, 128, "bf16", sides, sides, [[4] * 2], max_window=16)
    assert kv.scalekv_selftest_wait(20) == (1, 1)          # it runs out, and leaves the status raised
    assert kv.scalekv_selftest_wait(20) == (1, 1)          # so this one gives up at once: the CTA's other warps have to see that too
    kv.close()
