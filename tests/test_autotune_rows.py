"""FFTSEG_FLAG_AUTOTUNE at lengths that run as Bluestein rows in one SM: the row
kernel is the one schedule of those lengths, so the flag takes it too (it asks
for the fastest schedule; it must not switch to the slower power-of-two rows)."""
import pytest

import siggen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1407_6915_gb300 as fs  # noqa: E402


@pytest.mark.parametrize("n", [2049, 10007, 12288 - 1])
def test_autotune_takes_the_row_kernel(n):
    x = torch.from_numpy(siggen.uniform(5300 + n, 3 * n).reshape(3, n)).cuda()
    default, tuned = fs.Plan(n, 3), fs.Plan(n, 3, flags=fs.FLAG_AUTOTUNE)
    assert tuned.info() == default.info()
    assert torch.equal(tuned.exec(x), default.exec(x))
    # power-of-two rows are still what FLAG_BLUESTEIN asks for
    both = fs.Plan(n, 3, flags=fs.FLAG_AUTOTUNE | fs.FLAG_BLUESTEIN).info()
    assert both["n1"] == 1 << (2 * n - 2).bit_length()
