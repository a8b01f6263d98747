"""The radix sort's two forms, all digit passes in one launch and one launch per
pass: equal over sizes; and where the device refuses to run all tiles at once,
the passes are launched one by one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_12392_gb300 import rcp  # noqa: E402

pytestmark = pytest.mark.gpu

TILE = 7168


def _check(n, bits, resident_tiles):
    rng = np.random.default_rng(n + bits)
    keys = rng.integers(0, 1 << bits, n, dtype=np.uint32)
    dk = torch.from_numpy(keys.view(np.int32).copy()).cuda()
    dv = torch.arange(n, dtype=torch.int32, device="cuda")
    rcp.rcp_debug_sort_pairs_tiles(dk, dv, n, bits, resident_tiles, torch.cuda.current_stream())
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(dk.cpu().numpy().view(np.uint32), keys[order])
    assert np.array_equal(dv.cpu().numpy(), order)


@pytest.mark.parametrize("n", [2, 1000, TILE, TILE + 1, 30_000, 300_001])
@pytest.mark.parametrize("bits", [8, 30])
@pytest.mark.parametrize("resident_tiles", [0, -1])
def test_both_forms(n, bits, resident_tiles):
    _check(n, bits, resident_tiles)


@pytest.mark.parametrize("bits", [8, 30])
def test_more_tiles_than_the_device_runs_at_once(bits):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    _check((sms + 3) * TILE + 5, bits, 1 << 20)
    torch.cuda.synchronize()  # and no error is left behind
    _check(20_000, bits, -1)
