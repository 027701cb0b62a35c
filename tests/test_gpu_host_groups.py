"""Host-buffer calls whose samples are cut into the path's own channel groups (of at
least 32 MB): a short last group, groups of unequal time splits, rows that need
padding, checked 8-bit channels, against the device-buffer call; and a caller's
chan_group, which stands.  Integer results: equal."""
import pytest
import torch

from test_gpu_correlate import mw  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,N,C,T,kw,groups", [
    (4, 64, 101, 20000, {}, 4),                   # 27 channels a group, 20 in the last
    (4, 250, 70, 4001, {}, 3),                    # rows padded on the device
    (8, 96, 75, 6000, {}, 3),                     # longer than one exact segment
    (8, 250, 5, 20000, {}, 2),                    # few items: groups split in time
    (8, 96, 75, 6000, dict(kind=1), 3),
    (4, 64, 101, 20000, dict(chan_group=50), 3),
    (4, 64, 101, 20000, dict(chan_group=101), 1),
    (4, 64, 101, 20000, dict(mma_shape=1), 4),
])
def test_host_groups(mw, bits, N, C, T, kw, groups):  # noqa: F811
    gen = torch.Generator().manual_seed(N + C)
    volt = torch.randint(0, 256, (C * T * N * (bits // 4),), dtype=torch.uint8, generator=gen)
    if bits == 8:
        volt[volt == 128] = 0  # -8 and -128 are outside the range
    else:
        volt[(volt & 15) == 8] = 0
        volt[(volt >> 4) == 8] = 0
    host = volt.pin_memory()
    p = mw.Plan(N, C, T, bits, **kw)
    ref = p.correlate(volt.cuda())
    out = torch.empty(ref.shape, dtype=ref.dtype).pin_memory()
    p.set_timing(True)
    p.correlate_host(host, out)
    assert p.status() == 0
    assert p.timing().h2d_copies == groups
    assert torch.equal(out, ref.cpu())
    p.close()
