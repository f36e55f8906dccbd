"""Merged launches on the GPU: a program that gdag_issue merges gives what its
launches give one by one (the serial policy merges nothing), at the sizes
where the merged kernels can go wrong."""
import numpy as np
import pytest
import torch

import datagen
from paper_2012_09646_gb300 import gdag as G
from paper_2012_09646_gb300.workloads import BsDag, ImgDag, MlDag, VecDag, gaussian_weights

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


def run_ml(policy, rows, feats, k1, k2, X, T1, b1, T2, b2):
    """Two score launches over one X (each its own classes); the scores."""
    with G.Context(policy=policy) as ctx:
        dev = [torch.as_tensor(np.ascontiguousarray(t)).cuda() for t in (X, T1, b1, T2, b2)]
        a = [ctx.array(t) for t in dev]
        S = [torch.full((rows, k), -1.0, device="cuda") for k in (k1, k2)]
        s = [ctx.array(t) for t in S]
        torch.cuda.synchronize()
        p = ctx.program()
        p.launch("dense_scores", a[0], a[1], a[2], s[0], rows, feats, k1)
        p.launch("dense_scores", a[0], a[3], a[4], s[1], rows, feats, k2)
        n = launches(ctx, p.issue)
        return [t.clone() for t in S], n


# the tensor-core pair: one row, the tile's edges, more tiles than SMs; one
# stage per team and the longest rows; class counts that differ.  The CUDA-core
# halves: both forms, one padded width.  Last: forms that stay apart
@pytest.mark.parametrize("rows,feats,k1,k2,want", [
    (1, 64, 10, 10, 1), (127, 128, 1, 10, 1), (128, 1024, 10, 3, 1), (129, 192, 7, 10, 1), (19457, 64, 10, 10, 1),
    (20000, 1024, 9, 10, 1), (1, 32, 10, 9, 1), (4097, 96, 12, 10, 1), (300, 992, 12, 12, 1), (301, 992, 16, 13, 1),
    (100, 128, 10, 11, 2), (100, 96, 12, 8, 2)])
@pytest.mark.parametrize("values", ["recipe", "general", "wide"])
def test_two_score_launches_equal_single_ones(rows, feats, k1, k2, want, values):
    g = np.random.default_rng(rows + feats)
    X, T1, b1, _, _ = datagen.ml_inputs(rows, feats=feats, classes=k1, seed=1)
    _, _, _, T2, b2 = datagen.ml_inputs(rows, feats=feats, classes=k2, seed=2)
    if values == "general":  # tables whose three pieces are all needed
        T1, T2 = (g.normal(0, 1, t.shape).astype(np.float32) for t in (T1, T2))
        X = g.integers(-256, 257, X.shape).astype(np.int32)
    if values == "wide":     # integers that bfloat16 cannot hold, in the first and last rows
        X = X.copy()
        X[0, 0], X[-1, -1] = 257, -70000
    merged, n = run_ml(G.GDAG_POLICY_PARALLEL, rows, feats, k1, k2, X, T1, b1, T2, b2)
    single, m = run_ml(G.GDAG_POLICY_SERIAL_ASYNC, rows, feats, k1, k2, X, T1, b1, T2, b2)
    assert (n, m) == (want, 2)
    for a, b in zip(merged, single):
        assert same_bits(a, b)


@pytest.mark.parametrize("rows,classes,want", [(1, 1, 1), (127, 2, 1), (129, 10, 1), (1000, 16, 1), (513, 17, 1),
                                               (4097, 32, 1), (32768, 10, 1), (32769, 10, 3)])
@pytest.mark.parametrize("swap", [False, True])
def test_softmaxes_and_labels_equal_their_launches(rows, classes, want, swap):
    g = np.random.default_rng(rows)
    S = [(g.normal(0, 9, (rows, classes)) + 0.0).astype(np.float32) for _ in range(2)]
    S[0][0, :] = S[1][0, :] = 0.0                    # ties: the lowest class
    if rows > 100:
        S[0][5, 0], S[1][7, classes - 1] = np.nan, np.inf
    got = []
    for policy in (G.GDAG_POLICY_PARALLEL, G.GDAG_POLICY_SERIAL_ASYNC):
        with G.Context(policy=policy) as ctx:
            t = [torch.from_numpy(s.copy()).cuda() for s in S]
            lab = torch.full((rows,), -1, dtype=torch.int32, device="cuda")
            a = [ctx.array(x) for x in t]
            L = ctx.array(lab)
            torch.cuda.synchronize()
            p = ctx.program()
            for x in (a[::-1] if swap else a):
                p.launch("row_softmax", x, rows, classes)
            p.launch("argmax_combine", a[0], a[1], L, rows, classes)
            n = launches(ctx, p.issue)
            assert n == (want if policy == G.GDAG_POLICY_PARALLEL else 3)
            got.append([x.clone() for x in t] + [lab.clone()])
    for a, b in zip(got[0][:2], got[1][:2]):
        assert same_bits(torch.nan_to_num(a, nan=7.0), torch.nan_to_num(b, nan=7.0))
    assert torch.equal(got[0][2], got[1][2])


def test_ml_program_equals_its_launches():
    rows = 5000
    inp = datagen.ml_inputs(rows, feats=256, classes=10, seed=4)
    got = []
    for policy, want in ((G.GDAG_POLICY_PARALLEL, 2), (G.GDAG_POLICY_SERIAL_ASYNC, 5)):
        with G.Context(policy=policy) as ctx:
            m = MlDag(ctx, rows, 256, 10)
            m.load(*inp)
            for _ in range(3):
                assert launches(ctx, m.launch_all) == want
            got.append([t.clone() for t in (m.S1, m.S2, m.labels)])
    for a, b in zip(*got):
        assert torch.equal(a, b)
