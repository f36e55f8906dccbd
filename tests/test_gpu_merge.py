"""Merged launches on the GPU: a program that gdag_issue merges gives what its
launches give one by one (the serial policy merges nothing), at the sizes
where the merged kernels can go wrong."""
import numpy as np
import pytest
import torch

import datagen
from paper_2012_09646_gb300 import gdag as G
from paper_2012_09646_gb300.workloads import BsDag, ImgDag, VecDag, gaussian_weights

pytestmark = pytest.mark.gpu


def launches(ctx, fn):
    before = ctx.stats()["launches"]
    fn()
    ctx.sync()
    return ctx.stats()["launches"] - before


def same_bits(a, b):
    return torch.equal(a.view(torch.int32), b.view(torch.int32))


# one pixel; a single row and column; images narrower than a lane's four
# columns; both sides of a strip (112 and 120 columns) and of a band; odd
# widths; several strips and bands; tall and wide
@pytest.mark.parametrize("rows,cols", [(1, 1), (1, 9), (9, 1), (2, 3), (5, 6), (11, 111), (12, 112), (13, 113),
                                       (24, 120), (25, 121), (48, 449), (333, 225), (64, 2048), (2050, 64),
                                       (1031, 1027)])
@pytest.mark.parametrize("special", [False, True])
def test_img_program_equals_its_launches(rows, cols, special):
    img = datagen.image(rows, cols, seed=rows + cols).copy()
    if special:  # infinities and a NaN where their neighbourhoods reach edges
        img.flat[0] = np.inf
        img.flat[-1] = -np.inf
        img[rows // 2, cols // 2] = np.nan
    got = []
    for policy, want in ((G.GDAG_POLICY_PARALLEL, 1), (G.GDAG_POLICY_SERIAL_ASYNC, 10)):
        with G.Context(policy=policy) as ctx:
            d = ImgDag(ctx, rows, cols)
            d.img.copy_(torch.from_numpy(img.reshape(-1)))
            torch.cuda.synchronize()
            assert launches(ctx, d.launch_all) == want
            got.append([t.clone() for t in (d.b5, d.b9, d.s, d.mm5, d.mm9, d.e5, d.e9, d.out)])
    for a, b in zip(got[0][:7], got[1][:7]):
        assert same_bits(torch.nan_to_num(a, nan=7.0), torch.nan_to_num(b, nan=7.0))
        assert torch.equal(a.isnan(), b.isnan())
    # out is four products and sums of those: each rounds once, contracted or not
    a, b = got[0][7], got[1][7]
    fine = b.isfinite()
    assert torch.equal(fine, a.isfinite())
    assert (a[fine] - b[fine]).abs().max().item() <= 4 * 2.0 ** -24 * 4 * max(1.0, b[fine].abs().max().item()) \
        if fine.any() else True


@pytest.mark.parametrize("ra,rb,merged", [(1, 2, True), (1, 3, True), (1, 4, True), (2, 3, True), (3, 4, True),
                                          (2, 2, False), (4, 2, False), (2, 5, False)])
def test_img_program_radii(ra, rb, merged):
    rows, cols = 70, 243
    img = torch.from_numpy(datagen.image(rows, cols, seed=3).reshape(-1)).cuda()
    got = []
    for policy in (G.GDAG_POLICY_PARALLEL, G.GDAG_POLICY_SERIAL_ASYNC):
        with G.Context(policy=policy) as ctx:
            d = ImgDag(ctx, rows, cols)
            d.R5, d.R9 = ra, rb
            d.w5, d.w9 = gaussian_weights(ra, 1.0).cuda(), gaussian_weights(rb, 2.0).cuda()
            d.W5, d.W9 = ctx.array(d.w5), ctx.array(d.w9)
            d.img.copy_(img)
            torch.cuda.synchronize()
            n = launches(ctx, d.launch_all)
            assert n == (1 if merged and policy == G.GDAG_POLICY_PARALLEL else 10)
            got.append([t.clone() for t in (d.b5, d.b9, d.s, d.mm5, d.mm9, d.e5, d.e9)])
    for a, b in zip(*got):
        assert same_bits(a, b)


# no element and a tail only; one block and two; every block of the reduction
@pytest.mark.parametrize("n", [0, 1, 3, 5, 4096, 4097, 8191, 1_000_000, 5_000_003])
@pytest.mark.parametrize("swap", [False, True])
def test_vec_program_equals_its_launches(n, swap):
    x, y = datagen.vec_inputs(max(n, 1), seed=n)
    got = []
    for policy, want in ((G.GDAG_POLICY_PARALLEL, 1), (G.GDAG_POLICY_SERIAL_ASYNC, 3)):
        with G.Context(policy=policy) as ctx:
            v = VecDag(ctx, n)
            for _ in range(2):  # the reduction's arrival counter comes back to zero
                v.x.copy_(torch.from_numpy(x))
                v.y.copy_(torch.from_numpy(y))
                torch.cuda.synchronize()
                p = ctx.program()
                a, b = (v.Y, v.X) if swap else (v.X, v.Y)
                p.launch("vec_square", a, n)
                p.launch("vec_square", b, n)
                p.launch("vec_reduce_diff", v.X, v.Y, v.Z, v.S, n)
                assert launches(ctx, p.issue) == want
            got.append([t.clone() for t in (v.x, v.y, v.z)])
    for a, b in zip(*got):
        assert same_bits(a, b)


@pytest.mark.parametrize("off", [(0, 1), (1, 0), (1, 1)])
def test_vec_program_unaligned(off):
    n = 5001
    x, y = datagen.vec_inputs(n, seed=9)
    got = []
    for policy in (G.GDAG_POLICY_PARALLEL, G.GDAG_POLICY_SERIAL_ASYNC):
        with G.Context(policy=policy) as ctx:
            v = VecDag(ctx, n)
            bufs = [torch.zeros(n + 4, device="cuda") for _ in off]
            arrs = []
            for b, o, src in zip(bufs, off, (x, y)):
                b[o:o + n].copy_(torch.from_numpy(src))
                arrs.append(ctx.array(dev=b.data_ptr() + 4 * o, nbytes=4 * n))
            torch.cuda.synchronize()
            p = ctx.program()
            p.launch("vec_square", arrs[0], n)
            p.launch("vec_square", arrs[1], n)
            p.launch("vec_reduce_diff", arrs[0], arrs[1], v.Z, v.S, n)
            p.issue()
            ctx.sync()
            got.append([t.clone() for t in bufs])
            z = v.z.item()
            d = (x * x).astype(np.float64) - (y * y).astype(np.float64)
            assert abs(z - d.sum()) <= 1e-5 * np.abs(d).sum()
    for a, b in zip(*got):
        assert same_bits(a, b)


@pytest.mark.parametrize("n,count,want", [(1, 2, 1), (4099, 10, 1), (156_253, 32, 1), (156_253, 40, 2),
                                          (1 << 21, 3, 1), ((1 << 21) + 1, 3, 3)])
def test_bs_books_equal_their_launches(n, count, want):
    got = []
    for policy in (G.GDAG_POLICY_PARALLEL, G.GDAG_POLICY_SERIAL_ASYNC):
        with G.Context(policy=policy) as ctx:
            d = BsDag(ctx, n, count=count, host=False)
            d.load_device(datagen.bs_inputs(n, count=count, seed=n))
            k = launches(ctx, d.launch_all)
            assert k == (want if policy == G.GDAG_POLICY_PARALLEL else count)
            got.append([t.clone() for t in d.C])
    for a, b in zip(*got):
        assert same_bits(a, b)
