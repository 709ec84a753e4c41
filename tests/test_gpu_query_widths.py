"""Queries of every value width against the oracle, key by key: the window reads
differ with the width (aligned, moved, grouped over lanes), and the last warp of
a query is ragged."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2411_12365_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_12365_gb300 import burr  # noqa: E402


def _u32(t):
    a = t.cpu().numpy()
    return a.view(f"u{a.dtype.itemsize}").astype(np.uint32)


@pytest.mark.parametrize("mode", [burr.THRESH_2BIT, burr.THRESH_1PLUS])
@pytest.mark.parametrize("r", range(1, 33))
def test_every_width_matches_oracle(r, mode):
    for n in (1, 64, 9_001 if r != 8 else 160_001):   # one block, two, and more (r = 8: a table past 128 KB)
        keys = I.keys_torch(n, "cuda", seed=7 * r + n)
        vals = I.values_torch(keys, r)
        h = burr.build(keys, vals, r, threshold_mode=mode, partition_slots=1024, min_partition_slots=0)
        ref = O.build(keys.cpu().numpy().view(np.uint64), _u32(vals), r=r, threshold_mode=mode, partition_slots=1024,
                      min_partition_slots=0)
        assert ref.ok
        assert torch.equal(h.query(keys), vals)
        others = I.keys_torch(2_111, "cuda", offset=1 << 40)
        want = ref.query(others.cpu().numpy().view(np.uint64))
        for nq in (1, 3, 31, 32, 33, 257, 2_111):
            assert np.array_equal(_u32(h.query(others[:nq])), want[:nq]), (n, nq)


def test_no_bumping_layers():
    for r in (8, 16, 32, 3):
        keys = I.keys_torch(3_000, "cuda", seed=r)
        vals = I.values_torch(keys, r)
        h = burr.build(keys, vals, r, layers=0)
        assert torch.equal(h.query(keys[:1_001]), vals[:1_001])


@pytest.mark.parametrize("r,n", [(3, 300_000), (3, 4_400_000), (5, 150_000), (5, 900_000), (6, 800_000), (7, 320_000),
                                 (8, 9_001), (13, 180_000), (14, 320_000), (15, 150_000), (16, 80_000), (32, 40_000)])
def test_larger_tables_are_read_otherwise_and_equal(r, n):
    """Tables past the sizes at which a width changes its loads or leaves L1."""
    keys = I.keys_torch(n, "cuda", seed=r)
    vals = I.values_torch(keys, r)
    h = burr.build(keys, vals, r)
    ref = O.build(keys.cpu().numpy().view(np.uint64), _u32(vals), r=r)
    assert torch.equal(h.query(keys), vals)
    others = I.keys_torch(20_011, "cuda", offset=1 << 40)
    assert np.array_equal(_u32(h.query(others)), ref.query(others.cpu().numpy().view(np.uint64)))
