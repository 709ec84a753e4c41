"""Segments whose runs meet their stored run late or never: most buckets compare
masks that differ, which are then replaced.  Whole exports against the serial
oracle, and the same on every repetition."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_12365_gb300 import inputs as I
from tests.export_format import describe_difference

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_12365_gb300 import burr  # noqa: E402


@pytest.mark.parametrize("n,r,mode,alpha", [(250_007, 8, burr.THRESH_2BIT, 1.0), (250_007, 8, burr.THRESH_1PLUS, 0.98),
                                            (180_001, 20, burr.THRESH_1PLUS, 1.015)])
def test_late_meetings_are_repeatable(n, r, mode, alpha):
    keys = I.keys_torch(n, "cuda", seed=3 * n + r)
    vals = I.values_torch(keys, r)
    v = vals.cpu().numpy()
    ref = O.build(keys.cpu().numpy().view(np.uint64), v.view(f"u{v.dtype.itemsize}").astype(np.uint32), r=r,
                  threshold_mode=mode, alpha=alpha)
    assert ref.ok
    want = ref.export()
    for _ in range(4):
        got = burr.build(keys, vals, r, threshold_mode=mode, load_factor=alpha).export()
        assert got == want, describe_difference(got, want)
