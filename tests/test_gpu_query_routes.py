"""Queries on the other sides of the lines that choose a kernel: loads far from the
default, tables off 32-byte boundaries, few keys, one flag word.  Against the
oracle, key by key."""
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


def _check(h, ref, keys, vals):
    others = I.keys_torch(70_003, "cuda", offset=1 << 40)
    want = ref.query(others.cpu().numpy().view(np.uint64))
    for nq in (1, 33, 255, 256, 32_767, 32_768, 70_003):
        assert np.array_equal(_u32(h.query(others[:nq])), want[:nq]), nq
    assert torch.equal(h.query(keys), vals)


@pytest.mark.parametrize("mode", [burr.THRESH_2BIT, burr.THRESH_1PLUS])
@pytest.mark.parametrize("alpha", [0.8, 1.015, 1.3])
@pytest.mark.parametrize("r", [1, 2, 3, 4, 5, 6, 8, 12, 15, 16, 17, 20, 31, 32])
def test_loads_and_sizes(r, alpha, mode):
    for n in (3_000, 90_001):
        keys = I.keys_torch(n, "cuda", seed=r + n)
        vals = I.values_torch(keys, r)
        ref = O.build(keys.cpu().numpy().view(np.uint64), _u32(vals), r=r, threshold_mode=mode, alpha=alpha)
        _check(burr.build(keys, vals, r, threshold_mode=mode, load_factor=alpha), ref, keys, vals)


@pytest.mark.parametrize("mode", [burr.THRESH_2BIT, burr.THRESH_1PLUS])
@pytest.mark.parametrize("r", [1, 3, 8, 16, 20, 31, 32])
def test_tables_off_32_byte_boundaries(r, mode):
    keys = I.keys_torch(40_009, "cuda", seed=r)
    vals = I.values_torch(keys, r)
    ref = O.build(keys.cpu().numpy().view(np.uint64), _u32(vals), r=r, threshold_mode=mode)
    dev, shifted = torch.cuda.current_device(), {}

    def alloc(n, stream):
        p = torch.cuda.caching_allocator_alloc(n + 64, dev, stream)
        q = (p + 31) // 32 * 32 + 16
        shifted[q] = p
        return q

    burr.set_allocator(alloc, lambda ptr, stream: torch.cuda.caching_allocator_delete(shifted.pop(ptr)))
    h = None
    try:
        h = burr.build(keys, vals, r, threshold_mode=mode)
        _check(h, ref, keys, vals)
    finally:
        if h is not None:
            h.free()
        torch.cuda.synchronize()
        burr.set_allocator(None, None)
    assert not shifted
