"""The radix sort at the edges of its tiles (7,168 pairs) and beyond the tiles
that run at once, for each number of digit passes: bit-exact against a stable
sort."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 255, 7167, 7168, 7169, 14336, 14337, 8 * 7168 + 1, 1 << 20, 5_000_001])
@pytest.mark.parametrize("bits", [8, 16, 24, 30])
@pytest.mark.parametrize("spread", ["uniform", "few"])
def test_tiles_and_passes(n, bits, spread):
    rng = np.random.default_rng(n + bits)
    if spread == "uniform":
        keys = rng.integers(0, 1 << bits, n, dtype=np.uint32)
    else:  # nearly every key in two buckets of every digit
        keys = (rng.integers(0, 2, n, dtype=np.uint32) * np.uint32((1 << bits) - 1)) ^ (rng.random(n) < 1e-3)
        keys = keys.astype(np.uint32)
    order = np.argsort(keys, kind="stable")
    sorts = [rcp.rcp_debug_sort_pairs] + ([rcp.rcp_sort_pairs_static] if n <= rcp.rcp_sort_static_capacity() else [])
    for sort in sorts:
        dk = torch.from_numpy(keys.view(np.int32)).cuda()
        dv = torch.arange(n, dtype=torch.int32, device="cuda")
        sort(dk, dv, n, bits, torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert np.array_equal(dk.cpu().numpy().view(np.uint32), keys[order])
        assert np.array_equal(dv.cpu().numpy(), order)
