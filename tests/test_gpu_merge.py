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


# widths around the last columns that a strip's halo lanes hold (112 k + 4 and 112 k
# + 8): the edge maps' largest steps lie beside the left or the right edge, so a
# column taken wrongly there moves the range and with it e5, e9 and out
@pytest.mark.parametrize("cols", [224, 225, 227, 228, 229, 231, 232, 340, 344, 452, 1012, 4036])
@pytest.mark.parametrize("columns", [(-4, -1), (-1, None), (-8, -4), (1, 4), (0, 1), (4, 8)])
def test_img_range_beside_the_edges(cols, columns):
    rows = 8
    img = np.zeros((rows, cols), np.float32)
    img[:, slice(*columns)] = 1.0
    got = []
    for policy in (G.GDAG_POLICY_PARALLEL, G.GDAG_POLICY_SERIAL_ASYNC):
        with G.Context(policy=policy) as ctx:
            d = ImgDag(ctx, rows, cols)
            d.img.copy_(torch.from_numpy(img.reshape(-1)))
            torch.cuda.synchronize()
            d.launch_all()
            ctx.sync()
            got.append([t.clone() for t in (d.b5, d.b9, d.s, d.mm5, d.mm9, d.e5, d.e9)])
    for a, b in zip(*got):
        assert same_bits(a, b)


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


# one tile in all; more tiles than SMs in either; odd counts, so that a CTA's
# two teams end on different convolutions; a plain-store row width (w / 2 not a
# multiple of 8) beside a tensor-store one, both ways round; a partial tile
@pytest.mark.parametrize("a,b", [((1, 2, 8), (1, 2, 8)), ((1, 2, 64), (1, 4, 264)), ((1, 4, 264), (2, 6, 72)),
                                 ((2, 6, 72), (3, 66, 192)), ((5, 130, 128), (1, 2, 520)), ((3, 110, 256), (4, 90, 256))])
def test_two_convolutions_and_pools_equal_their_launches(a, b):
    g = np.random.default_rng(sum(a) * 31 + sum(b))
    bf = torch.bfloat16
    ins = []
    for n, h, w in (a, b):
        ins.append((torch.from_numpy(g.random((n, 3, h, w), dtype=np.float32)).to(bf),
                    torch.from_numpy(g.normal(0, 0.3, (64, 3, 3, 3)).astype(np.float32)).to(bf),
                    torch.from_numpy(g.normal(0, 0.1, 64).astype(np.float32))))
    got = []
    for policy, want in ((G.GDAG_POLICY_PARALLEL, 2), (G.GDAG_POLICY_SERIAL_ASYNC, 4)):
        with G.Context(policy=policy) as ctx:
            p, outs, keep = ctx.program(), [], []
            pools = []
            for (n, h, w), (x, wt, bias) in zip((a, b), ins):
                t = [v.cuda() for v in (x, wt, bias)]
                o = torch.full((n, 64, h // 2, w // 2), -1.0, dtype=bf, device="cuda")
                e = torch.full((n, 64), -1.0, device="cuda")
                st = torch.zeros(1, dtype=torch.int32, device="cuda")
                A = [ctx.array(v) for v in t + [o, st, e]]
                p.launch("conv3x3_relu_pool", A[0], A[1], A[2], A[3], A[4], n, h, w)
                pools.append((A[3], A[5], n * 64, (h // 2) * (w // 2)))
                outs += [o, e, st]
                keep += t + A
            for q in pools:
                p.launch("avgpool_global", *q)
            torch.cuda.synchronize()
            for _ in range(2):
                assert launches(ctx, p.issue) == want
            got.append([t.clone() for t in outs])
    for x, y in zip(*got):
        assert torch.equal(x.view(torch.int16) if x.dtype == bf else x, y.view(torch.int16) if y.dtype == bf else y)
    assert got[0][2].item() == 0 and got[0][5].item() == 0
    # the first convolution against plain float64
    (n, h, w), (x, wt, bias) = a, ins[0]
    ref = torch.nn.functional.conv2d(x.double(), wt.double(), bias.double(), padding=1).clamp_min(0)
    ref = torch.nn.functional.max_pool2d(ref, 2)
    assert (got[0][0].double().cpu() - ref).abs().max() <= 2.0 ** -8 * ref.abs().max()


# sizes that merge; one pair whose lengths differ; the empty vector
@pytest.mark.parametrize("n,nnz,m,mnz", [(1, 0, 1, 0), (500, 4000, 500, 4000), (3000, 0, 100, 9000), (1279, 1, 1281, 7),
                                         (60_000, 300_000, 20_000, 500_000), (0, 0, 50, 60)])
def test_two_products_norms_and_scalings_equal_their_launches(n, nnz, m, mnz):
    got = []
    for policy, want in ((G.GDAG_POLICY_PARALLEL, 3), (G.GDAG_POLICY_SERIAL_ASYNC, 6)):
        with G.Context(policy=policy) as ctx:
            p, outs, keep, tail = ctx.program(), [], [], []
            for k, (rows, nz) in enumerate(((n, nnz), (m, mnz))):
                g = np.random.default_rng(rows + nz)
                ends = np.sort(g.integers(0, rows + 1, nz)) if rows else np.zeros(0, np.int64)
                if rows and nz > 100:  # a row that spans many tiles
                    ends[nz // 4: 3 * nz // 4] = ends[nz // 2]
                rp = np.searchsorted(ends, np.arange(rows + 1), side="left").astype(np.int32)
                rp[-1] = nz if rows else 0
                col = g.integers(0, max(rows, 1), max(nz, 1)).astype(np.int32)
                val = g.normal(0, 1, max(nz, 1)).astype(np.float32)
                x = g.normal(0, 1, max(rows, 1)).astype(np.float32)
                t = [torch.from_numpy(v).cuda() for v in (rp, col, val, x)]
                y = torch.full((max(rows, 1),), 7.0, device="cuda")
                nrm = torch.full((1,), -1.0, device="cuda")
                sc = [torch.zeros(G.gdag_scratch_bytes(q, rows + nz), dtype=torch.uint8, device="cuda")
                      for q in ("spmv_partition", "spmv_csr", "l2norm")]
                A = [ctx.array(v) for v in t + [y, nrm] + sc]
                ctx.launch("spmv_partition", A[0], A[6], rows, nz)
                p.launch("spmv_csr", A[0], A[1], A[2], A[3], A[6], A[4], A[7], rows, nz)
                tail.append((A[4], A[5], A[8], rows))
                outs += [y, nrm]
                keep += t + sc + A
                if k == 0 and policy == G.GDAG_POLICY_PARALLEL and rows:
                    ref = np.zeros(rows)
                    np.add.at(ref, np.searchsorted(rp[1:], np.arange(nz), side="right"),
                              val[:nz].astype(np.float64) * x[col[:nz]])
                    mag = np.zeros(rows)
                    np.add.at(mag, np.searchsorted(rp[1:], np.arange(nz), side="right"),
                              np.abs(val[:nz].astype(np.float64) * x[col[:nz]]))
            for v, q, s, rows in tail:
                p.launch("l2norm", v, q, s, rows)
            for v, q, s, rows in tail:
                p.launch("scale", v, q, rows)
            ctx.sync()
            k = launches(ctx, p.issue)
            assert k == want
            got.append([t.clone() for t in outs])
    for a, b in zip(*got):
        assert same_bits(a, b)
    if n:
        y, nrm = got[0][0].double().cpu().numpy()[:n], got[0][1].item()
        assert abs(nrm - np.sqrt((ref ** 2).sum())) <= 1e-5 * max(nrm, 1e-30) + 1e-30
        # a product rounds once, a sum of up to 64 terms in a chain, the rest in
        # trees and per tile, the norm and the division once each: under 256 ulp
        # halves of the sum of |terms|
        if nrm > 0:
            assert (np.abs(y * nrm - ref) <= 2.0 ** -24 * 256 * mag + 1e-30).all()


# one plane row; images whose planes take the pools' scalar loads; more tiles and
# planes than the chip holds at a time
@pytest.mark.parametrize("n,h,w,classes,swap", [(1, 2, 8, 1, False), (3, 6, 24, 33, True), (2, 66, 264, 10, False),
                                                (40, 128, 256, 10, True)])
def test_dl_program_equals_its_launches(n, h, w, classes, swap):
    g = np.random.default_rng(n * h + w)
    bf = torch.bfloat16
    f = lambda *s: torch.from_numpy(g.normal(0, 0.3, s).astype(np.float32))  # noqa: E731
    ins = [(f(n, 3, h, w).to(bf), f(64, 3, 3, 3).to(bf), f(64)) for _ in range(2)]
    wd, bd = f(128, classes), f(classes)
    got = []
    for policy, want in ((G.GDAG_POLICY_PARALLEL, 1), (G.GDAG_POLICY_SERIAL_ASYNC, 5)):
        with G.Context(policy=policy) as ctx:
            x = [[t.cuda() for t in b] for b in ins]
            P = [torch.zeros((n, 64, h // 2, w // 2), dtype=bf, device="cuda") for _ in x]
            E = [torch.zeros((n, 64), device="cuda") for _ in x]
            st = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in x]
            dense = [wd.cuda(), bd.cuda(), torch.zeros((n, classes), device="cuda")]
            AX = [[ctx.array(t) for t in b] for b in x]
            AP, AE, AS, AD = ([ctx.array(t) for t in v] for v in (P, E, st, dense))
            p = ctx.program()
            for k in (0, 1):
                p.launch("conv3x3_relu_pool", *AX[k], AP[k], AS[k], n, h, w)
            for k in (1, 0) if swap else (0, 1):
                p.launch("avgpool_global", AP[k], AE[k], n * 64, (h // 2) * (w // 2))
            p.launch("concat_dense", AE[0], AE[1], *AD, n, 64, classes)
            out = []
            torch.cuda.synchronize()
            for step in range(3):  # other inputs each time: a stage that ran ahead would show
                assert launches(ctx, p.issue) == want
                out += [t.clone() for t in P + E + st + dense[2:]]
                for b in x:
                    b[0].mul_(-0.5)
                torch.cuda.synchronize()
            got.append(out)
    for a, b in zip(*got):
        assert torch.equal(a.view(torch.int16) if a.dtype == bf else a, b.view(torch.int16) if b.dtype == bf else b)


@pytest.mark.parametrize("late", [0, 1])
def test_a_unit_waits_for_parents_on_busy_streams(late):
    """The unit's inputs are made by kernels on two streams, one of them long, and
    its members' results are used on others at once."""
    n, m = 200_000, 10_000_000
    g = torch.Generator(device="cuda").manual_seed(3)
    S = [torch.rand(k, generator=g, device="cuda") * 90 + 10 for k in ((m, n) if late == 0 else (n, m))]
    got = []
    for policy, want in ((G.GDAG_POLICY_PARALLEL, 1), (G.GDAG_POLICY_SERIAL_ASYNC, 3)):
        with G.Context(policy=policy) as ctx:
            v = VecDag(ctx, n)
            SA = [ctx.array(s) for s in S]
            C = [torch.zeros_like(s) for s in S]
            CA = [ctx.array(c) for c in C]
            use = [ctx.array(t) for t in (torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda"))]
            keep = []
            torch.cuda.synchronize()
            for step in range(4):
                for k, dst in ((0, v.X), (1, v.Y)):
                    for _ in range(6):
                        ctx.launch("bs_call", SA[k], CA[k], S[k].numel(), 60.0 + step, 0.1, 0.2, 1.0)
                    # the first n prices into the unit's array, after all of them
                    ctx.launch("unsharp", ctx.array(C[k][:n]), CA[k], dst, 0.0, n)
                p = ctx.program()
                p.launch("vec_square", v.X, n)
                p.launch("vec_square", v.Y, n)
                p.launch("vec_reduce_diff", v.X, v.Y, v.Z, v.S, n)
                before = ctx.stats()["launches"]
                p.issue()
                assert ctx.stats()["launches"] - before == want
                for a, b in zip((v.X, v.Y), use):
                    ctx.launch("unsharp", a, a, b, 0.0, n)
                ctx.sync()
                keep += [t.clone() for t in (v.x, v.y, v.z, use[0].tensor, use[1].tensor)]
            got.append(keep)
    for a, b in zip(*got):
        assert same_bits(a, b)
    assert not torch.equal(got[0][0], got[0][5])  # the steps differ
