"""An allocation that finds the device full gets the buffers that another context keeps."""
import pytest

from paper_1112_5280_gb300 import lqcd

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def test_a_full_device_takes_back_what_other_contexts_keep():
    import torch

    one, two = lqcd.Context(0), lqcd.Context(0)
    kept = [one.field((16, 16, 16, 32), "f64") for _ in range(40)]  # 25.2 MB each
    for f in kept:
        f.close()
    torch.cuda.synchronize()
    # 512 MiB are left: less than the field below needs (805 MB), more with one's buffers
    rest = torch.empty(torch.cuda.mem_get_info()[0] - 512 * MIB, dtype=torch.uint8, device="cuda")
    f = two.field((32, 32, 32, 64), "f64")
    assert f.nbytes == 32 ** 3 * 64 * 24 * 8 and f.norm2() == 0.0
    f.close()
    del rest
    torch.cuda.empty_cache()
    one.close()
    two.close()
