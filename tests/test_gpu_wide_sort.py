"""The radix sort on both sides of the size from which it takes the wide passes, and just above it
with runs of equal and of consecutive keys: exactly numpy's stable argsort."""
import numpy as np
import pytest
import torch

from gpu_common import renderer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(1 << 20) - 1, 1 << 20, (1 << 20) + 8193, 3_700_001])
@pytest.mark.parametrize("bits,runs", [((0, 31), False), ((16, 29), True), ((0, 9), False)])
def test_radix_sort_around_the_wide_size(n, bits, runs):
    rng = np.random.default_rng(n)
    keys = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
    if runs:
        keys = ((np.arange(n) // 7 * 2654435761 % (1 << 13) + np.arange(n) % 7) << 16 |
                np.arange(n) % 65521).astype(np.uint32)
    vals = np.arange(n, dtype=np.uint32)
    k, v = (torch.from_numpy(x.view(np.int32).copy()).cuda() for x in (keys, vals))
    r = renderer()
    r.ctx.radix_sort_u32(k.data_ptr(), v.data_ptr(), n, *bits, r.stream_handle())
    torch.cuda.synchronize()
    digit = (keys >> np.uint32(bits[0])) & np.uint32((1 << (bits[1] - bits[0])) - 1)
    order = np.argsort(digit, kind="stable")
    np.testing.assert_array_equal(v.cpu().numpy().view(np.uint32), vals[order])
    np.testing.assert_array_equal(k.cpu().numpy().view(np.uint32), keys[order])
