"""Which copies may run beside kernels of their context (recording backend, CPU
only): those are left to the copy engines; and the host's check that one
pinned allocation holds a view."""
import pathlib
import subprocess

from paper_2012_09646_gb300 import gdag as G

ROOT = pathlib.Path(__file__).resolve().parent.parent


def test_range_within_an_allocation(tmp_path):
    exe = tmp_path / "host_range"
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-Werror", "-I",
                    str(ROOT / "paper_2012_09646_gb300" / "csrc"), str(ROOT / "tests" / "c" / "host_range.cpp"),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def copies(ctx):
    """(node, beside) of the copies issued, in order."""
    return [(o.node, o.beside) for o in G.gdag_ops_export(ctx.h)
            if o.type in (G.GDAG_OP_COPY_H2D, G.GDAG_OP_COPY_D2H)]


def make(**kw):
    ctx = G.Context(backend="fake", record_log=True, **kw)
    return ctx, [ctx.array(dev=(i + 1) << 24, nbytes=400) for i in range(4)]


def test_copies_beside_kernels():
    ctx, (x, y, z, w) = make()
    ctx.write(x)                       # nothing runs
    ctx.write(y)                       # beside a copy only
    ctx.launch("vec_square", x, 100)   # on x's stream
    ctx.write(x)                       # follows the kernel on its stream
    ctx.write(z)                       # beside it
    ctx.prefetch_host(w)               # beside it
    ctx.launch("vec_square", y, 100)   # a kernel on a second stream
    ctx.write(x)                       # follows one, beside the other
    assert [b for _, b in copies(ctx)] == [0, 0, 0, 1, 1, 1]
    ctx.sync()
    ctx.write(z)                       # everything known to be complete
    assert copies(ctx)[-1][1] == 0
    ctx.close()


def test_copies_of_a_step_that_the_host_reads():
    """Write, write, compute, read: no copy of it is beside a kernel, step after step."""
    ctx, (x, y, z, w) = make(retire_by_query=True)
    sc = ctx.array(dev=9 << 24, nbytes=G.gdag_scratch_bytes("vec_reduce_diff", 100))
    p = ctx.program()
    p.write(x)
    p.write(y)
    p.launch("vec_square", x, 100)
    p.launch("vec_square", y, 100)
    p.launch("vec_reduce_diff", x, y, z, sc, 100)
    for _ in range(5):
        p.issue()
        ctx.read(z, None, 0, 4)
    assert len(copies(ctx)) == 15 and not any(b for _, b in copies(ctx))
    ctx.close()


def test_serial_policies_have_one_stream():
    ctx, (x, y, _, _) = make(policy=G.GDAG_POLICY_SERIAL_ASYNC)
    ctx.launch("vec_square", x, 100)
    ctx.write(y)
    assert copies(ctx) == [(1, 0)]
    ctx.close()


def test_copies_beside_several_copies():
    """Copies by kernels share the link; those by an engine come one after another, so
    that what follows the first overlaps the others: from the third on, by an engine."""
    ctx, a = make()
    a += [ctx.array(dev=(i + 9) << 24, nbytes=400) for i in range(4)]
    for x in a:
        ctx.write(x)
    assert [b for _, b in copies(ctx)] == [0, 0] + [1] * 6
    ctx.sync()
    ctx.write(a[0])
    assert copies(ctx)[-1][1] == 0
    ctx.close()
