"""Batches of one long structure and many short ones, banded in segments: the
scratch follows the sum of the partitions' lengths, not the longest one's times
their number, and every export equals the structure's own build."""
import numpy as np
import pytest

from paper_2411_12365_gb300 import inputs as I
from tests.export_format import describe_difference

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_12365_gb300 import burr  # noqa: E402


def _inputs(sizes, r, seed=3):
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    keys = I.keys_torch(int(offs[-1]), "cuda", seed=seed)
    return keys, I.values_torch(keys, r), offs


def _model_bytes(sizes, r, alpha=1.015):
    """Device bytes of a build by the server's admission model, less its constant term."""
    vb = 1 if r <= 8 else (2 if r <= 16 else 4)
    n = np.asarray(sizes, dtype=np.float64)
    m = n / alpha + 128
    return float((n * (8 + vb) * 4 + m * (8 + vb) * 2 + m / 64 * r * 8).sum())


@pytest.mark.parametrize("kw", [dict(partition_slots=1 << 22, min_partition_slots=1 << 22), dict(layers=0)])
def test_scratch_of_one_long_structure_among_many_short_ones(kw):
    sizes, r = [100] * 600 + [4_000_000] + [100] * 400, 8
    keys, vals, offs = _inputs(sizes, r)
    dev, live, peak = torch.cuda.current_device(), {}, [0]

    def alloc(n, stream):
        p = torch.cuda.caching_allocator_alloc(n, dev, stream)
        live[p] = n
        peak[0] = max(peak[0], sum(live.values()))
        return p

    def free(ptr, stream):
        del live[ptr]
        torch.cuda.caching_allocator_delete(ptr)

    burr.set_allocator(alloc, free)
    try:
        hs = burr.build_batch(keys, vals, offs, [r] * len(sizes), **kw)
        got = hs[600].export()
        burr.free_all(hs)
        torch.cuda.synchronize()
    finally:
        burr.set_allocator(None, None)
    assert not live
    assert peak[0] <= _model_bytes(sizes, r) + (32 << 20), peak[0]
    want = burr.build(keys[60_000:4_060_000].clone(), vals[60_000:4_060_000].clone(), r, **kw).export()
    assert got == want, describe_difference(got, want)


@pytest.mark.parametrize("mode", [burr.THRESH_2BIT, burr.THRESH_1PLUS])
@pytest.mark.parametrize("r,kw", [(8, {}), (20, dict(cut_search=burr.CUT_DIFF)), (3, dict(layers=0)),
                                  (8, dict(partition_slots=1 << 14, lower_partition_slots=1 << 13, load_factor=1.1,
                                           cut_search=burr.CUT_MINBUMP)),
                                  (16, dict(partition_slots=8_320, min_partition_slots=0))])
def test_mixed_lengths_equal_single_builds(r, kw, mode):
    # partitions just too short for two segments, ragged ones, and long ones, in no order
    sizes = [100, 8_100, 300_011, 1, 8_400, 0, 70_003, 64, 12_345] + [200] * 50 + [150_000]
    keys, vals, offs = _inputs(sizes, r, seed=r)
    hs = burr.build_batch(keys, vals, offs, [r] * len(sizes), threshold_mode=mode, **kw)
    for s, h in enumerate(hs):
        if 10 < s < 58:
            continue
        a, b = int(offs[s]), int(offs[s + 1])
        got, want = h.export(), burr.build(keys[a:b], vals[a:b], r, threshold_mode=mode, **kw).export()
        assert got == want, (s, describe_difference(got, want))


def test_launches_of_a_segmented_base_case_are_counted():
    # 32-bucket segments: 1 + ceil(190 / 32) passes and the last one, instead of one launch
    def launches(n):
        keys, vals, offs = _inputs([n], 8)
        st = burr.build_batch(keys, vals, offs, [8], layers=0)[0].stats()
        assert st["fallback_attempt"] == 0
        return st["kernel_launches"]

    assert launches(200_000) - launches(5_000) == 1 + -(-190 // 32) + 1 - 1


def test_searched_cuts_choose_the_back_substitution_of_plain_ones():
    # partitions of 32 to 47 blocks (the last ones): past the size up to which blocks are reduced first
    # (50,000 slots per block of the longest), but within that of partitions 32 blocks longer
    keys, vals, offs = _inputs([1_500_000, 1_500_000], 8)

    def stats(cut):
        st = burr.build_batch(keys, vals, offs, [8, 8], cut_search=cut, layers=1, partition_slots=2_048,
                              min_partition_slots=2_048)[0].stats()
        assert st["fallback_attempt"] == 0
        return st["kernel_launches"]

    assert stats(burr.CUT_DIFF) - stats(burr.CUT_NONE) == 1   # the search
