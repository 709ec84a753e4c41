"""The band sweep where it can go wrong: more rows than registers (loads far
above one), partitions banded in segments, more rows in a bucket than are staged at once, buckets of one
block's worth of slots, values that travel inside the row keys (up to 16 bits)
and beside them (17 and more), in both threshold modes.  Whole exports against
the serial oracle, bit for bit."""
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

B64 = dict(bucket_slots=64, levels=(0, 16, 40, 64))
CASES = [
    (20_011, 8, 0.5, {}),                          # sparse: empty blocks
    (20_011, 16, 1.45, {}), (20_011, 17, 1.5, {}),   # around 192 rows per bucket
    (30_000, 32, 3.0, {}), (30_000, 1, 12.0, {}),  # most rows bumped, layer after layer
    (15_013, 8, 1.015, B64), (15_013, 24, 2.5, B64),
    (127, 8, 1.015, {}), (130, 16, 1.015, {}), (64, 32, 1.0, {}),
    (40_000, 8, 1.015, dict(partition_slots=128, min_partition_slots=0)),   # a cut at every bucket
    # few long partitions, banded in segments: just too short, one bucket past two segments, odd
    # lengths, both value layouts, searched cuts, loads where segments seldom or never meet again
    (8_030, 8, 1.015, {}), (8_290, 8, 1.015, {}), (300_011, 24, 1.015, {}), (270_007, 16, 1.015, {}),
    (400_003, 5, 1.015, dict(partition_slots=16384, cut_search=burr.CUT_DIFF)),
    (150_000, 8, 0.97, {}), (150_000, 9, 1.1, {}), (200_000, 32, 1.6, {}), (120_000, 8, 0.9, dict(layers=0)),
    (260_003, 7, 1.02, dict(partition_slots=40_960, lower_partition_slots=8192)), (90_001, 8, 1.015, B64),
]


@pytest.mark.parametrize("mode", [burr.THRESH_2BIT, burr.THRESH_1PLUS])
@pytest.mark.parametrize("n,r,alpha,kw", CASES)
def test_sweep_matches_oracle(n, r, alpha, kw, mode):
    keys = I.keys_torch(n, "cuda", seed=n + r)
    vals = I.values_torch(keys, r)
    got = burr.build(keys, vals, r, threshold_mode=mode, load_factor=alpha, **kw).export()
    v = vals.cpu().numpy()
    names = {"bucket_slots": "B"}
    ref = O.build(keys.cpu().numpy().view(np.uint64), v.view(f"u{v.dtype.itemsize}").astype(np.uint32), r=r,
                  threshold_mode=mode, alpha=alpha, **{names.get(k, k): x for k, x in kw.items()})
    assert ref.ok
    want = ref.export()
    assert got == want, describe_difference(got, want)


@pytest.mark.parametrize("r,mode,cut,alpha", [(8, burr.THRESH_2BIT, burr.CUT_NONE, 1.015),
                                              (3, burr.THRESH_1PLUS, burr.CUT_DIFF, 1.015),
                                              (1, burr.THRESH_2BIT, burr.CUT_MINBUMP, 1.6)])
def test_packed_records_match_oracle(r, mode, cut, alpha):
    """Layers sorted in two passes with one-byte values: records and values travel
    packed; just past the smallest such layer, whole exports against the oracle."""
    n = int(8_400_000 * alpha) + 101
    keys = I.keys_torch(n, "cuda", seed=r)
    vals = I.values_torch(keys, r)
    got = burr.build(keys, vals, r, threshold_mode=mode, cut_search=cut, load_factor=alpha).export()
    ref = O.build(keys.cpu().numpy().view(np.uint64), vals.cpu().numpy().astype(np.uint32), threads=16, r=r,
                  threshold_mode=mode, cut_search=cut, alpha=alpha)
    assert ref.ok
    want = ref.export()
    assert got == want, describe_difference(got, want)
