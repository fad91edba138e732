"""The block that an LJ pass on full lists runs with: at most 256 threads; FP64
with a warp per atom halves it while the grid has less than two blocks per SM
of the device in use; the mixed path keeps the caller's block."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [128, 256, 512])
def test_block_follows_the_device(block):
    import torch
    from paper_2511_22951_gb300 import _build
    _build.build()
    f = ctypes.CDLL(_build.LIB)._ZN3mdk8lj_blockEiiii
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    top = min(block, 256)
    for tpa in (1, 2, 4, 8, 32):
        for n in (0, 1, 256, 2 * sms - 1, 2 * sms, 4 * sms - 1, 4 * sms, 8 * sms, 16 * sms, 10 ** 6):
            assert f(1, n, tpa, block) == top
            got = f(0, n, tpa, block)
            if tpa < 32:
                assert got == top
            else:
                want = [b for b in (256, 128, 64, 32) if b <= top and n * 32 // b >= 2 * sms]
                assert got == (want[0] if want else 32)
