"""The sort does not depend on how long its blocks wait for one another."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2601_20429_gb300 import native as N


@pytest.mark.parametrize("max_waits", [0, 1, 3])
@pytest.mark.parametrize("n,bits", [(1025, 64), (30_000, 13), (262_145, 64), (1_500_000, 64)])
def test_sort_with_short_waits(n, bits, max_waits):
    """Blocks that stop waiting at once count the keys before them: still numpy's stable order, each time."""
    rng = np.random.default_rng(n)
    keys = rng.integers(0, 1 << 63, n, dtype=np.uint64)
    keys[: n // 2] &= np.uint64(0xFF00FF)                 # digits that most of a tile shares
    part = keys & np.uint64((1 << bits) - 1) if bits < 64 else keys
    order = np.argsort(part, kind="stable")
    for _ in range(3):
        k, v = torch.from_numpy(keys.view(np.int64).copy()).cuda(), torch.arange(n, dtype=torch.int32, device="cuda")
        temp = N.grtx_sort_pairs_bounded(k, v, max_waits, bits)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(v.cpu().numpy(), order)
        np.testing.assert_array_equal(k.cpu().numpy().view(np.uint64), keys[order])
        del temp


def test_negative_wait_is_refused():
    k, v = torch.zeros(4, dtype=torch.int64, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda")
    with pytest.raises(N.GrtxError):
        N.grtx_sort_pairs_bounded(k, v, -1)
