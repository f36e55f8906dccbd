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


# around the limit of copies in one-byte pieces
@pytest.mark.parametrize("off", [1, 2, 4, 12])
@pytest.mark.parametrize("nbytes", [(64 << 10) - 4, (64 << 10), (64 << 10) + 4])
def test_unaligned_copies(off, nbytes):
    with G.Context() as ctx:
        dev = torch.zeros(nbytes + 64, dtype=torch.uint8, device="cuda")
        a = ctx.array(dev, host=torch.empty(nbytes + 64, dtype=torch.uint8, pin_memory=True))
        data = np.random.default_rng(off).integers(0, 256, nbytes).astype(np.uint8)
        ctx.write(a, data, off, nbytes)
        ctx.sync()
        want = np.zeros(nbytes + 64, np.uint8)
        want[off:off + nbytes] = data
        assert np.array_equal(dev.cpu().numpy(), want)
        dev.add_(1)
        torch.cuda.synchronize()
        b = ctx.array(dev, host=torch.full((nbytes + 64,), 9, dtype=torch.uint8, pin_memory=True))
        ctx.read(b, None, off, nbytes)
        got = b.host.numpy()
        assert np.array_equal(got[off:off + nbytes], data + np.uint8(1))
        assert (got[:off] == 9).all() and (got[off + nbytes:] == 9).all()


def test_views_inside_a_registered_buffer():
    """Memory that the caller pinned by registration: views at its start, inside and at
    its end."""
    size = 1 << 20
    raw = np.zeros(size + (64 << 10), np.uint8)
    skip = -raw.ctypes.data % (64 << 10)
    buf = torch.from_numpy(raw[skip:skip + size])
    rt = torch.cuda.cudart()
    torch.zeros(1, device="cuda")
    assert int(rt.cudaHostRegister(buf.data_ptr(), size, 0)) == 0
    try:
        with G.Context() as ctx:
            for lo, hi in ((0, 4096), (777, 5000), (size - 1000, size), (0, size)):
                buf.copy_(torch.randint(0, 256, (size,), dtype=torch.uint8))
                dev = torch.zeros(hi - lo, dtype=torch.uint8, device="cuda")
                a = ctx.array(dev, host=buf[lo:hi])
                ctx.write(a)
                ctx.sync()
                assert torch.equal(dev.cpu(), buf[lo:hi])
                ctx.unregister(a)
    finally:
        rt.cudaHostUnregister(buf.data_ptr())
