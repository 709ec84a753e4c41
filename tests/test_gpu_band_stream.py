"""Sparse layers, whose rows are inserted as a stream: whole exports against the
serial oracle over value widths, bucket sizes, cuts, both threshold modes, packed
records and base cases, and batches and shards of them."""
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
from paper_2411_12365_gb300 import shard  # noqa: E402

B64 = dict(bucket_slots=64, levels=(0, 16, 40, 64))
CASES = [
    (20_011, 8, 0.5, dict(partition_slots=1_024, min_partition_slots=0)),
    (300_007, 17, 0.25, dict(partition_slots=4_096)),
    (100_003, 1, 0.7, dict(partition_slots=128, min_partition_slots=0)),
    (200_003, 32, 0.85, dict(partition_slots=1_024, cut_search=burr.CUT_DIFF)),
    (150_011, 16, 0.6, dict(partition_slots=512, min_partition_slots=0, **B64)),
    (60_001, 24, 0.9, dict(partition_slots=128, min_partition_slots=0, **B64)),
    (1_500_007, 8, 0.92, dict(partition_slots=2_048, min_partition_slots=2_048)),   # a split launch's bound on parts
    (64, 8, 0.3, {}), (1, 32, 0.5, {}), (2_000, 9, 0.94, {}),
    (3_001, 8, 1.015, dict(layers=0, fallback_slack=1.0)), (5_003, 16, 1.015, dict(layers=0, fallback_slack=0.2)),
    (4_400_003, 8, 0.5, {}), (7_000_003, 3, 0.8, dict(partition_slots=1_024, cut_search=burr.CUT_MINBUMP)),   # packed
]


@pytest.mark.parametrize("mode", [burr.THRESH_2BIT, burr.THRESH_1PLUS])
@pytest.mark.parametrize("n,r,alpha,kw", CASES)
def test_stream_matches_oracle(n, r, alpha, kw, mode):
    keys = I.keys_torch(n, "cuda", seed=n + r)
    vals = I.values_torch(keys, r)
    got = burr.build(keys, vals, r, threshold_mode=mode, load_factor=alpha, **kw).export()
    v = vals.cpu().numpy()
    names = {"bucket_slots": "B", "fallback_slack": "fb_slack"}
    ref = O.build(keys.cpu().numpy().view(np.uint64), v.view(f"u{v.dtype.itemsize}").astype(np.uint32), threads=16, r=r,
                  threshold_mode=mode, alpha=alpha, **{names.get(k, k): x for k, x in kw.items()})
    assert ref.ok
    want = ref.export()
    assert got == want, describe_difference(got, want)


@pytest.mark.parametrize("mode", [burr.THRESH_2BIT, burr.THRESH_1PLUS])
@pytest.mark.parametrize("kw", [dict(load_factor=0.6), dict(load_factor=0.85, cut_search=burr.CUT_DIFF, partition_slots=2_048),
                                dict(layers=0, fallback_slack=0.8)])
def test_sparse_batches_equal_single_builds(kw, mode):
    sizes = [100, 20_011, 1, 0, 70_003, 64, 5_000] + [300] * 40 + [1_000_003]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    keys = I.keys_torch(int(offs[-1]), "cuda", seed=5)
    vals = I.values_torch(keys, 8)
    hs = burr.build_batch(keys, vals, offs, [8] * len(sizes), threshold_mode=mode, **kw)
    for s in (0, 1, 2, 3, 4, 5, 6, 7, 46, 47):
        a, b = int(offs[s]), int(offs[s + 1])
        got, want = hs[s].export(), burr.build(keys[a:b], vals[a:b], 8, threshold_mode=mode, **kw).export()
        assert got == want, (s, describe_difference(got, want))


def test_sparse_shards_equal_the_single_build():
    n, kw = 400_003, dict(load_factor=0.5, partition_slots=4_096)
    keys = I.keys_torch(n, "cuda", seed=1)
    vals = I.values_torch(keys, 8)
    want = burr.build(keys, vals, 8, **kw).export()
    got = shard.build_sharded_virtual([keys[g::3].contiguous() for g in range(3)], [vals[g::3].contiguous() for g in range(3)], 8, **kw)
    assert got == want, describe_difference(got, want)


def test_window_of_a_test_is_an_error_here_too():
    keys = I.keys_torch(300_000, "cuda", seed=1)
    vals = I.values_torch(keys, 8)
    with pytest.raises(burr.BurrError) as e:
        burr.build(keys, vals, 8, load_factor=0.6, partition_slots=1_024, flags=burr.FLAG_TEST_WINDOW)
    assert e.value.code == burr.ERR_INTERNAL


def test_time_falls_with_the_load():
    """A layer of a quarter of the keys in as many slots takes much less time to band."""
    def band_ms(n, alpha):
        keys = I.keys_torch(n, "cuda", seed=2)
        vals = I.values_torch(keys, 8)
        return min(burr.build(keys, vals, 8, load_factor=alpha, partition_slots=4_096, min_partition_slots=4_096,
                              flags=burr.FLAG_TIMING).stats()["stage_ms"][0][1] for _ in range(5))

    assert band_ms(5_000_000, 0.25) < 0.6 * band_ms(20_000_000, 1.0)   # 0.26 / 1.0 ms; both swept 1.0
