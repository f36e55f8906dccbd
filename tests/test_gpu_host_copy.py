"""Host writes and reads of every route (a kernel for short copies of pinned
views, the copy engines for the rest): the bytes arrive, and no others change,
for offsets and sizes around the kernels' piece sizes and their limit."""
import numpy as np
import pytest
import torch

from paper_2012_09646_gb300 import gdag as G

pytestmark = pytest.mark.gpu
LIMIT = 4 << 20


@pytest.mark.parametrize("view", ["pinned", "pageable", "library"])
@pytest.mark.parametrize("off,nbytes", [(0, 1), (0, 15), (0, 16), (0, 17), (3, 40), (4, 4), (4, 4099), (16, 62500),
                                        (1, 4097), (0, LIMIT - 1), (0, LIMIT), (16, LIMIT + 1), (5, LIMIT)])
def test_write_and_read_move_exactly_their_bytes(view, off, nbytes):
    size = off + nbytes + 64
    g = np.random.default_rng(nbytes)
    with G.Context() as ctx:
        dev = torch.full((size,), 7, dtype=torch.uint8, device="cuda")
        host = None
        if view != "library":
            host = torch.empty(size, dtype=torch.uint8, pin_memory=view == "pinned")
        a = ctx.array(dev, host=host)
        for _ in range(3):  # new bytes in the same view each time
            data = g.integers(0, 256, nbytes).astype(np.uint8)
            ctx.write(a, data, off, nbytes)
            ctx.sync()
            want = np.full(size, 7, np.uint8)
            want[off:off + nbytes] = data
            assert np.array_equal(dev.cpu().numpy(), want)
        # a device-side change, read back over a marked view
        dev.add_(1)
        torch.cuda.synchronize()
        b = ctx.array(dev, host=torch.full((size,), 9, dtype=torch.uint8, pin_memory=view == "pinned")
                      if view != "library" else None)
        out = np.zeros(nbytes, np.uint8)
        ctx.read(b, out, off, nbytes)
        assert np.array_equal(out, data + np.uint8(1))
        if view != "library":
            assert (b.host[:off] == 9).all() and (b.host[off + nbytes:] == 9).all()
